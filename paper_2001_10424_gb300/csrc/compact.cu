// compact.cu - operator products between compact vectors in one kernel.
//
// Through the padded layout a product is four launches (clear, pack, stencil,
// unpack) that move seven vectors; here a block loads the compact entries of
// its tile with a one-face halo into shared memory (faces that are not
// unknowns read as 0 and cost no memory access), forms the rows there and
// writes the compact result: two vectors and one launch. What then bounds a
// large product is the FP64 pipe (8.75 operations per 2D unknown), a small one
// the launch and the wait for it. 1023 x 770: 86.5 -> 48 us, 130 x 95 x 77:
// 156 -> 139 us, 64 x 64 without a handle 34 -> 24 us per call, host side
// included. The rows are those of k_mac_tile (same operations and order).
#include "compact.cuh"

#include <algorithm>
#include <type_traits>

#include "../../include/gkb.h"
#include "kernels_impl.cuh"
#include "prof.h"
#include "solver.cuh"

namespace gkb {

namespace {

constexpr int C3B = 3;    // blocks of the 3D kernel per SM

// W row over wscale at a face of component C, position p: the links of w_row
// in its order, with the neighbours from nb(axis, direction)
template <int C, int DIM, class F>
__device__ __forceinline__ double links(const Lvl& L, const int (&p)[3], double xf, F nb) {
  const double mu = L.mu0;
  double acc = 0.0;
  if (p[C] < L.n[C]) acc = fma(mu, xf - nb(C, 1), acc);
  if (p[C] > 0) acc = fma(mu, xf - nb(C, -1), acc);
  const double area = face_half<C>(L, p) ? 0.5 : 1.0;
#pragma unroll
  for (int A = 0; A < DIM; ++A) {
    if (A == C) continue;
    if (p[A] + 1 < L.n[A]) acc = fma(area * mu, xf - nb(A, 1), acc);
    else if (!L.nat[2 * A + 1]) acc = fma(2.0 * area * mu, xf, acc);
    if (p[A] > 0) acc = fma(area * mu, xf - nb(A, -1), acc);
    else if (!L.nat[2 * A]) acc = fma(2.0 * area * mu, xf, acc);
  }
  return acc;
}

// y = M x (wonly: W x). Tile of CTX x TY positions; in 3D the block walks kz
// planes with rings of four planes of x and three of divergences in shared
// memory (one plane more than the rows read, so that two barriers a plane
// suffice), the next plane's entries fetched while the current one is computed.
template <int DIM, int CTX, int TY>
__global__ void __launch_bounds__(256, DIM == 3 ? C3B : 4) k_op_compact(const __grid_constant__ Lvl L, const __grid_constant__ Compact c,
                                                                        int wonly, int kz,
                                                                       const double* __restrict__ x,
                                                                       double* __restrict__ y) {
  constexpr int NS = DIM == 3 ? 4 : 1, ND = DIM == 3 ? 3 : 1, W = CTX + 2, H = TY + 2, EN = DIM * W * H, NE = (EN + 255) / 256;
  __shared__ double X[NS][DIM][H][W];              // position (i0 - 1 + col, j0 - 1 + row)
  __shared__ double Dv[ND][TY + 1][CTX + 1];  // cell (i0 - 1 + col, j0 - 1 + row)
  const int tid = threadIdx.x, tx = tid % CTX, ty = tid / CTX;
  const int i0 = blockIdx.x * CTX, j0 = blockIdx.y * TY;
  const int k0 = DIM == 3 ? blockIdx.z * kz : 0, k1 = DIM == 3 ? min(k0 + kz, L.n[2] + L.nat[5]) : 1;
  const bool gd = L.has_gd && !wonly;
  auto slot = [](int k) { return DIM == 3 ? (k + 4) & 3 : 0; };
  auto dslot = [](int k) { return DIM == 3 ? (k + 3) % 3 : 0; };
  // this thread's entries of a plane: offset in x of plane lo_z of the
  // component, step per plane, planes that hold unknowns
  long long off[NE];
  int step[NE], kl[NE], kh[NE];
  double pre[NE];
#pragma unroll
  for (int e = 0; e < NE; ++e) {
    const int t = tid + e * 256, q = t / (W * H), r = (t - q * W * H) / W, col = t - (q * H + r) * W;
    const int i = i0 - 1 + col, j = j0 - 1 + r;
    kl[e] = 1;
    kh[e] = 0;
    off[e] = 0;
    step[e] = 0;
    if (t < EN && i >= c.lo[q][0] && i < c.lo[q][0] + c.ext[q][0] && j >= c.lo[q][1] && j < c.lo[q][1] + c.ext[q][1]) {
      kl[e] = c.lo[q][2];
      kh[e] = c.lo[q][2] + c.ext[q][2] - 1;
      step[e] = c.ext[q][0] * c.ext[q][1];
      off[e] = c.base[q] + (long long)(j - c.lo[q][1]) * c.ext[q][0] + (i - c.lo[q][0]);
    }
  }
  auto fetch = [&](int k) {
#pragma unroll
    for (int e = 0; e < NE; ++e)
      pre[e] = (k >= kl[e] && k <= kh[e]) ? __ldg(x + off[e] + (long long)(k - kl[e]) * step[e]) : 0.0;
  };
  auto commit = [&](int k) {
    double* s = &X[slot(k)][0][0][0];
#pragma unroll
    for (int e = 0; e < NE; ++e)
      if (tid + e * 256 < EN) s[tid + e * 256] = pre[e];
  };
  auto div_plane = [&](int k) {  // negative divergences of cell plane k, 0 outside the domain
    const int s0 = slot(k), s1 = slot(k + 1);
    for (int t = tid; t < (TY + 1) * (CTX + 1); t += 256) {
      const int r = t / (CTX + 1), q = t - r * (CTX + 1);
      double d = 0.0;
      if (cell_in(L, i0 - 1 + q, j0 - 1 + r, k)) {
        d = X[s0][0][r][q] - X[s0][0][r][q + 1] + X[s0][1][r][q] - X[s0][1][r + 1][q];
        if constexpr (DIM == 3) d += X[s0][2][r][q] - X[s1][2][r][q];
      }
      Dv[dslot(k)][r][q] = d;
    }
  };
  if constexpr (DIM == 3) {
    fetch(k0 - 1);
    commit(k0 - 1);
    fetch(k0);
    commit(k0);
    fetch(k0 + 1);
    if (gd) {
      __syncthreads();
      div_plane(k0 - 1);
    }
  } else {
    fetch(0);
    commit(0);
    __syncthreads();
  }
  for (int k = k0; k < k1; ++k) {
    if constexpr (DIM == 3) {
      commit(k + 1);
      if (k + 1 < k1) fetch(k + 2);
      __syncthreads();
    }
    if (gd) {
      div_plane(k);
      __syncthreads();
    }
    const int sc = slot(k), su = slot(k + 1), sd = slot(k - 1), dc = dslot(k), dd = dslot(k - 1);
#pragma unroll
    for (int rr = 0; rr < TY * CTX / 256; ++rr) {
      const int r = ty + 256 / CTX * rr, i = i0 + tx, j = j0 + r;
      const int p[3] = {i, j, k};
      auto face = [&](auto comp, double dm) {
        constexpr int C = decltype(comp)::value;
        if (!face_active<C>(L, i, j, k)) return;
        auto nb = [&](int axis, int dir) -> double {
          if (axis == 0) return X[sc][C][r + 1][tx + 1 + dir];
          if (axis == 1) return X[sc][C][r + 1 + dir][tx + 1];
          return X[dir > 0 ? su : sd][C][r + 1][tx + 1];
        };
        const double xf = X[sc][C][r + 1][tx + 1], dp = gd ? Dv[dc][r + 1][tx + 1] : 0.0;
        double v;
        if (const_regular<C>(L, p)) {
          double acc = nb(0, 1) + nb(0, -1) + nb(1, 1) + nb(1, -1);
          if constexpr (DIM == 3) acc += nb(2, 1) + nb(2, -1);
          v = const_row<double, 1>(L, 0.0, xf, acc, gd, dp, dm);
        } else {
          v = wall_row<double>(links<C, DIM>(L, p, xf, nb), L.wscale, gd, L.g2, dp, dm);
        }
        y[c.base[C] + ((long long)(k - c.lo[C][2]) * c.ext[C][1] + (j - c.lo[C][1])) * c.ext[C][0] +
          (i - c.lo[C][0])] = v;
      };
      face(std::integral_constant<int, 0>{}, gd ? Dv[dc][r + 1][tx] : 0.0);
      face(std::integral_constant<int, 1>{}, gd ? Dv[dc][r][tx + 1] : 0.0);
      if constexpr (DIM == 3) face(std::integral_constant<int, 2>{}, gd ? Dv[dd][r + 1][tx + 1] : 0.0);
    }
  }
}

// y = A p, one thread per position: its face of every component
template <int DIM>
__global__ void __launch_bounds__(256) k_grad_compact(const Lvl L, const Compact c, const double* __restrict__ p,
                                                       double* __restrict__ y) {
  const int i = blockIdx.x * 32 + threadIdx.x, j = blockIdx.y * 8 + threadIdx.y, k = blockIdx.z;
  auto cell = [&](int a, int b, int d) -> double {
    return cell_in(L, a, b, d) ? __ldg(p + ((long long)d * L.n[1] + b) * L.n[0] + a) : 0.0;
  };
  const double pc = cell(i, j, k);
  auto face = [&](auto comp, double pm) {
    constexpr int C = decltype(comp)::value;
    if (face_active<C>(L, i, j, k))
      y[c.base[C] + ((long long)(k - c.lo[C][2]) * c.ext[C][1] + (j - c.lo[C][1])) * c.ext[C][0] + (i - c.lo[C][0])] =
          L.ascale * (pc - pm);
  };
  face(std::integral_constant<int, 0>{}, cell(i - 1, j, k));
  face(std::integral_constant<int, 1>{}, cell(i, j - 1, k));
  if constexpr (DIM == 3) face(std::integral_constant<int, 2>{}, cell(i, j, k - 1));
}

// y = A^T x, one thread per cell
template <int DIM>
__global__ void __launch_bounds__(256) k_negdiv_compact(const Lvl L, const Compact c, const double* __restrict__ x,
                                                         double* __restrict__ y) {
  const int i = blockIdx.x * 32 + threadIdx.x, j = blockIdx.y * 8 + threadIdx.y, k = blockIdx.z;
  if (!cell_in(L, i, j, k)) return;
  auto at = [&](auto comp, int a, int b, int d) -> double {
    constexpr int C = decltype(comp)::value;
    if (!face_active<C>(L, a, b, d)) return 0.0;
    return __ldg(x + c.base[C] + ((long long)(d - c.lo[C][2]) * c.ext[C][1] + (b - c.lo[C][1])) * c.ext[C][0] +
                 (a - c.lo[C][0]));
  };
  std::integral_constant<int, 0> U;
  std::integral_constant<int, 1> V;
  double s = at(U, i, j, k) - at(U, i + 1, j, k) + at(V, i, j, k) - at(V, i, j + 1, k);
  if constexpr (DIM == 3) {
    std::integral_constant<int, 2> Wc;
    s += at(Wc, i, j, k) - at(Wc, i, j, k + 1);
  }
  y[((long long)k * L.n[1] + j) * L.n[0] + i] = L.ascale * s;
}

}  // namespace

void apply_compact(const Lvl& L, int op, const double* x, double* y, cudaStream_t s) {
  const Compact c = make_compact(L);
  const dim3 blk(32, 8);
  if (op == GKB_OP_W || op == GKB_OP_M) {
    ProfScope ps_(GKB_KC_APPLY, s, lvl_unknowns(L));
    const int wonly = op == GKB_OP_W;
    // positions that hold a face: n along an axis, n + 1 if the high side is natural
    const unsigned nx = L.n[0] + L.nat[1], ny = L.n[1] + L.nat[3], nz = L.dim == 3 ? L.n[2] + L.nat[5] : 1;
    auto up = [](unsigned a, unsigned b) { return (a + b - 1) / b; };
    if (L.dim == 2) {
      k_op_compact<2, 32, 16><<<dim3(up(nx, 32), up(ny, 16)), 256, 0, s>>>(L, c, wonly, 1, x, y);
    } else {
      // 16 x 16 tiles (160^3: 424 us, 32 x 8 tiles 468 us) unless the wide ones
      // waste 10 % fewer positions (a warp with few of them still takes its
      // full time on the FP64 pipe); eight planes per block where
      // that leaves four waves of blocks, two where four leave SMs empty, else
      // four (every block adds two planes of loads and one of divergences, but
      // a last wave that fills a third of the chip costs more)
      const bool wide = 11 * up(nx, 32) * 32 * up(ny, 8) * 8 < 10 * up(nx, 16) * 16 * up(ny, 16) * 16;
      const unsigned gx = wide ? up(nx, 32) : up(nx, 16), gy = wide ? up(ny, 8) : up(ny, 16);
      const unsigned kz = gx * gy * up(nz, 8) >= 4 * 152 * C3B ? 8 : gx * gy * up(nz, 4) >= 152 ? 4 : 2;
      const dim3 g(gx, gy, up(nz, kz));
      if (wide) k_op_compact<3, 32, 8><<<g, 256, 0, s>>>(L, c, wonly, (int)kz, x, y);
      else k_op_compact<3, 16, 16><<<g, 256, 0, s>>>(L, c, wonly, (int)kz, x, y);
    }
  } else if (op == GKB_OP_A) {
    ProfScope ps_(GKB_KC_LAYOUT, s, lvl_unknowns(L));
    if (L.dim == 2) k_grad_compact<2><<<face_grid(L), blk, 0, s>>>(L, c, x, y);
    else k_grad_compact<3><<<face_grid(L), blk, 0, s>>>(L, c, x, y);
  } else {
    ProfScope ps_(GKB_KC_LAYOUT, s, lvl_unknowns(L));
    if (L.dim == 2) k_negdiv_compact<2><<<cell_grid(L), blk, 0, s>>>(L, c, x, y);
    else k_negdiv_compact<3><<<cell_grid(L), blk, 0, s>>>(L, c, x, y);
  }
  GKB_CUDA(cudaGetLastError());
}

}  // namespace gkb
