// legs.cuh - one level's whole share of a 2D V-cycle as two kernels: the down
// leg (pre-smoothing, residual, restriction) and the up leg (prolongation,
// post-smoothing).
//
// As separate launches a level with smoother degree g costs 4 g + 5 kernels,
// each reading and writing whole vectors; below 512^2 a launch is mostly the
// kernel boundary (1.0 us of a 1.1 us FP32 launch inside a graph). Here a
// block owns a TW x TH tile of cells, loads the right-hand side (and the
// iterate and coarse correction) of the tile plus a halo into shared memory
// once, runs every step there on a region that shrinks by the step's radius,
// and writes only what leaves the level: the iterate of its tile and the
// restricted residual of its coarse faces. The halo costs recomputation
// instead of memory traffic and kernel boundaries.
//
// Every value is formed by the operations, in the order, of the separate
// launches (k_mac_tile, k_cheb2, the transfer kernels), so that both forms of
// a V-cycle agree bit for bit.
#pragma once
#include <type_traits>

#include "kernels_impl.cuh"

namespace gkb {

constexpr int LEG_NT = 256;      // threads per block
constexpr int LEG_MAX_DEG = 3;   // smoother degrees with an instance

template <typename T>
struct LegArgs {
  Lvl L, Lc;
  const T* b;     // right-hand side; with rd: the gathered part rU of it
  const T* rd;    // gathered slopes rD still to be transposed into b, or null
  T* bfull;       // down leg, with rd: receives the complete right-hand side
  T* xpre;        // the iterate after pre-smoothing (down: out, up: in)
  const T* xc;    // up: the coarse level's solution
  T* xout;        // up: the iterate after post-smoothing (not xpre)
  T* bc;          // down: rU of the coarse level
  T* tmp;         // down: rD of the coarse level
  const T* table; // class stencils
  T ca[LEG_MAX_DEG], cb[LEG_MAX_DEG];
  Fold2In<T> fs[LEG_MAX_DEG];  // interior stencils scaled by ca[k]
};

// tile geometry: halo cells below / above the owned cells on both axes. The
// residual is needed two cells below the tile (restriction), every smoothing
// step after the first needs two more on each side, the first one.
template <int DEG, int TW, int TH>
struct DownTile {
  static constexpr int HL = 2 * DEG + 2, HH = 2 * DEG;
  static constexpr int EW = TW + HL + HH, EH = TH + HL + HH, EN = EW * EH;
};
template <int DEG, int TW, int TH>
struct UpTile {
  static constexpr int HL = 2 * DEG, HH = 2 * DEG;
  static constexpr int EW = TW + HL + HH, EH = TH + HL + HH, EN = EW * EH;
};
// shared planes: b, x, r, d of both components; FP64 also the divergences,
// formed once per cell (the FP64 pipe is what it runs out of first)
template <typename T> struct LegPlanes { static constexpr int n = sizeof(T) == 8 ? 9 : 8; };
// the class stencils, 49 classes x 2 components x 7, follow the planes, then
// the scaled interior ones of every step: near a side every position has its
// own, and from global memory they would put an L2 round trip into every step
constexpr int LEG_FOLD = (FOLD2_CLASSES + LEG_MAX_DEG) * 14;

// entry t of that table
template <typename T>
__device__ __forceinline__ T leg_fold_entry(const LegArgs<T>& A, int t) {
  const int pc = t / 14, q = t - pc * 14;
  if (pc >= FOLD2_CLASSES) return A.fs[pc - FOLD2_CLASSES].c[q / 7][q % 7];
  return GKB_LDG(A.table + FOLD3_OFF + pc * 48 + (q < 7 ? q : 9 + q));
}
template <typename T, class G>
constexpr size_t leg_smem() { return ((size_t)LegPlanes<T>::n * G::EN + LEG_FOLD) * sizeof(T); }

// (C r) at tile offset o by the 7-point stencil f (fold2_apply's order; faces
// that are not unknowns hold 0, so their coefficients need no test)
template <typename T, int C, int EW, class Coef>
__device__ __forceinline__ T leg_fold(const T* ru, const T* rv, int o, Coef f) {
  T acc = mul_rn(f(0), C == 0 ? ru[o] : rv[o]);
  T v[6];
  if (C == 0) {
    v[0] = ru[o - EW]; v[1] = rv[o - 1]; v[2] = rv[o];
    v[3] = ru[o + EW]; v[4] = rv[o + EW - 1]; v[5] = rv[o + EW];
  } else {
    v[0] = ru[o - EW]; v[1] = ru[o]; v[2] = rv[o - 1];
    v[3] = ru[o + 1 - EW]; v[4] = ru[o + 1]; v[5] = rv[o + 1];
  }
#pragma unroll
  for (int u = 0; u < 6; ++u) acc = fma(f(1 + u), v[u], acc);
  return acc;
}

template <typename T>
struct Pair { T u, v; };

// the box [ia, ib] x [ja, jb] lies in blocks that take the scaled stencils
// (which makes every face in it active and every row regular)
__device__ __forceinline__ bool leg_inner(const Lvl& L, int ia, int ib, int ja, int jb) {
  return ia >= 0 && ja >= 0 && cheb2_scaled(L, ia, ja) && cheb2_scaled(L, ib, jb);
}

// shared state of a leg: the tile's planes and its place in the level
template <typename T, class G>
struct Leg {
  static constexpr int EW = G::EW, EH = G::EH, EN = G::EN;
  T *bu, *bv, *xu, *xv, *ru, *rv, *du, *dv, *D, *fold;
  int ei, ej, nx, ny, tid;
  bool inner;  // every position whose row or stencil is formed is an interior one

  __device__ __forceinline__ Leg(const Lvl& L, int i0, int j0, T* sm) {
    bu = sm; bv = bu + EN; xu = bv + EN; xv = xu + EN; ru = xv + EN; rv = ru + EN; du = rv + EN; dv = du + EN;
    D = dv + EN;
    fold = bu + LegPlanes<T>::n * EN;
    ei = i0 - G::HL;
    ej = j0 - G::HL;
    nx = L.n[0];
    ny = L.n[1];
    tid = threadIdx.x + blockDim.x * threadIdx.y;
    inner = leg_inner(L, ei, ei + EW - 1, ej, ej + EH - 1);
  }
  __device__ __forceinline__ bool act_u(int i, int j) const { return i >= 1 && i < nx && j >= 0 && j < ny; }
  __device__ __forceinline__ bool act_v(int i, int j) const { return i >= 0 && i < nx && j >= 1 && j < ny; }

  // the class stencils into shared memory (tiles near a side only)
  __device__ __forceinline__ void load_fold(const LegArgs<T>& A) const {
    if (inner) return;
    for (int t = tid; t < LEG_FOLD; t += LEG_NT) fold[t] = leg_fold_entry(A, t);
  }

  // put(tile offset, f(tile offset, i, j)) over the tile shrunk by S on every
  // side, a few positions of a thread at a time: all of them are evaluated
  // before the first is stored, so that their shared loads overlap
  template <int S, class F, class P>
  __device__ __forceinline__ void over(F f, P put) const {
    constexpr int RW = EW - 2 * S, RH = EH - 2 * S, N = RW * RH, TRIPS = (N + LEG_NT - 1) / LEG_NT;
    constexpr int U = TRIPS <= 4 ? TRIPS : (TRIPS + 1) / 2 <= 4 ? (TRIPS + 1) / 2 : 3;
    for (int t0 = tid; t0 < N; t0 += U * LEG_NT) {
      Pair<T> z[U];
      int o[U];
#pragma unroll
      for (int k = 0; k < U; ++k) {
        const int t = t0 + k * LEG_NT;
        const int r = t / RW, c = t - r * RW;
        o[k] = (r + S) * EW + c + S;
        if (t < N) z[k] = f(o[k], ei + S + c, ej + S + r);
      }
#pragma unroll
      for (int k = 0; k < U; ++k)
        if (t0 + k * LEG_NT < N) put(o[k], z[k]);
    }
  }

  // r = b - M x on the tile shrunk by S (0 on faces that are not unknowns)
  template <int S>
  __device__ __forceinline__ void residual(const Lvl& L) const {
    const bool gd = L.has_gd;
    if (sizeof(T) == 8 && gd) {
      over<S - 1>([&](int o, int, int) { return Pair<T>{xu[o] - xu[o + 1] + xv[o] - xv[o + EW], (T)0}; },
                  [&](int o, const Pair<T>& z) { D[o] = z.u; });
      __syncthreads();
    }
    auto div = [&](int o) -> T {
      if (sizeof(T) == 8) return D[o];
      return xu[o] - xu[o + 1] + xv[o] - xv[o + EW];
    };
    const T g2 = Kc<T>::g2(L), mu = Kc<T>::mu0(L), ws = Kc<T>::ws(L);
    over<S>([&](int o, int i, int j) {
      const T d0 = gd ? div(o) : (T)0;
      auto face = [&](const T* x, const T* b, T dm, bool act, bool reg, int sc, int st, bool hi, bool lo) -> T {
        if (!inner && !act) return (T)0;
        const T xf = x[o];
        if (inner || reg) {
          const T acc = x[o + 1] + x[o - 1] + x[o + EW] + x[o - EW];
          return const_row<T, 0>(L, b[o], xf, acc, gd, d0, dm);
        }
        // a face beside a wall of its tangential axis (w_row's links)
        T w = fma(mu, xf - x[o + sc], (T)0);
        w = fma(mu, xf - x[o - sc], w);
        w = hi ? fma((T)2 * mu, xf, w) : fma(mu, xf - x[o + st], w);
        w = lo ? fma((T)2 * mu, xf, w) : fma(mu, xf - x[o - st], w);
        return b[o] - wall_row<T>(w, ws, gd, g2, d0, dm);
      };
      return Pair<T>{
          face(xu, bu, gd ? div(o - 1) : (T)0, act_u(i, j), j >= 1 && j <= ny - 2, 1, EW, j == ny - 1, j == 0),
          face(xv, bv, gd ? div(o - EW) : (T)0, act_v(i, j), i >= 1 && i <= nx - 2, EW, 1, i == nx - 1, i == 0)};
    }, [&](int o, const Pair<T>& z) {
      ru[o] = z.u;
      rv[o] = z.v;
    });
    __syncthreads();
  }

  // one Chebyshev step on the tile shrunk by S: d = ca C r + cb d, x += d
  // (ZERO: x = d); FIRST: without the previous d
  template <int S, bool ZERO, bool FIRST>
  __device__ __forceinline__ void cheb(const LegArgs<T>& A, int k, const T* su, const T* sv) const {
    const T ca = A.ca[k], cb = A.cb[k];
    over<S>([&](int o, int i, int j) {
      Pair<T> z{(T)0, (T)0};
      if (inner) {
        z.u = leg_fold<T, 0, EW>(su, sv, o, [&](int q) { return A.fs[k].c[0][q]; });
        z.v = leg_fold<T, 1, EW>(su, sv, o, [&](int q) { return A.fs[k].c[1][q]; });
        if (!FIRST) {
          z.u = fma(cb, du[o], z.u);
          z.v = fma(cb, dv[o], z.v);
        }
      } else if (i >= 0 && i < nx && j >= 0 && j < ny) {
        const bool sc = cheb2_scaled(A.L, i, j);
        const T* f = fold + (sc ? FOLD2_CLASSES + k : cls7(i, nx) * 7 + cls7(j, ny)) * 14;
        const T zu = leg_fold<T, 0, EW>(su, sv, o, [&](int q) { return f[q]; });
        const T zv = leg_fold<T, 1, EW>(su, sv, o, [&](int q) { return f[7 + q]; });
        if (i >= 1) z.u = cheb_wall<T>(sc ? (T)1 : ca, zu, cb, FIRST ? (T)0 : du[o], FIRST);
        if (j >= 1) z.v = cheb_wall<T>(sc ? (T)1 : ca, zv, cb, FIRST ? (T)0 : dv[o], FIRST);
      }
      return z;
    }, [&](int o, const Pair<T>& z) {
      du[o] = z.u;
      dv[o] = z.v;
      xu[o] = ZERO ? z.u : xu[o] + z.u;
      xv[o] = ZERO ? z.v : xv[o] + z.v;
    });
    __syncthreads();
  }

  // the owned faces of the tile, f(tile offset, padded index of (i, j), i, j)
  template <int TW, int TH, class F>
  __device__ __forceinline__ void owned(const Lvl& L, F f) const {
    for (int t = tid; t < TW * TH; t += LEG_NT) {
      const int r = t / TW, c = t - r * TW;
      const int i = ei + G::HL + c, j = ej + G::HL + r;
      if (i < nx && j < ny) f((r + G::HL) * EW + c + G::HL, j * L.P + i, i, j);
    }
  }
};

// the restriction's gather at the coarse face whose lower fine face is at tile
// offset o (restrict_flux_gather's terms and order): r, q the residual of the
// face's and the other component, sn / st the strides along the face's normal
// and tangential axis
template <typename T>
__device__ __forceinline__ void leg_gather(const T* r, const T* q, int o, int sn, int st, T& rU, T& rD) {
  T su = 0, sd = 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int on = o + (k == 0 ? 0 : k == 1 ? sn : -sn);
    const T w = (k == 0) ? (T)1 : (T)0.5;
    const T lo = r[on], hi = r[on + st];
    su += w * (lo + hi);
    sd += w * (hi - lo);
  }
  sd += (T)-0.5 * (q[o + st] + q[o + st + sn]);
  sd += (T)0.5 * (q[o + st - 2 * sn] + q[o + st - sn]);
  rU = su;
  rD = sd;
}

// the coarse correction on coarse cell (I, J)'s 2 x 2 fine u and v faces
// (prolong_flux2d_body): u (0,0) (0,1) (1,0) (1,1), then v (0,0) (1,0) (0,1) (1,1)
template <typename T>
__device__ __forceinline__ void leg_correction(const Lvl& Lc, const T* GKB_RESTRICT xc, int I, int J, T (&e)[8]) {
#pragma unroll
  for (int q = 0; q < 8; ++q) e[q] = (T)0;
  if (I < 0 || I >= Lc.n[0] || J < 0 || J >= Lc.n[1]) return;
  const T du0 = coarse_slope<T, 0>(Lc, xc, I, J), du1 = coarse_slope<T, 0>(Lc, xc, I + 1, J);
  const T dv0 = coarse_slope<T, 1>(Lc, xc, I, J), dv1 = coarse_slope<T, 1>(Lc, xc, I, J + 1);
  const T u0 = coarse_face<T, 0>(Lc, xc, I, J, 0), u1 = coarse_face<T, 0>(Lc, xc, I + 1, J, 0);
  const T v0 = coarse_face<T, 1>(Lc, xc, I, J, 0), v1 = coarse_face<T, 1>(Lc, xc, I, J + 1, 0);
  const T ulo0 = u0 - du0, uhi0 = u0 + du0, ulo1 = u1 - du1, uhi1 = u1 + du1;
  const T vlo0 = v0 - dv0, vhi0 = v0 + dv0, vlo1 = v1 - dv1, vhi1 = v1 + dv1;
  const T fu = (T)0.5 * (dv1 - dv0), fv = (T)0.5 * (du1 - du0);
  if (I >= 1) {
    e[0] = ulo0;
    e[1] = uhi0;
  }
  e[2] = (T)0.5 * (ulo0 + ulo1) + fu;
  e[3] = (T)0.5 * (uhi0 + uhi1) + fu;
  if (J >= 1) {
    e[4] = vlo0;
    e[5] = vhi0;
  }
  e[6] = (T)0.5 * (vlo0 + vlo1) + fv;
  e[7] = (T)0.5 * (vhi0 + vhi1) + fv;
}

// x = smooth(0, b) from zero, r = b - M x, (bc, tmp) = the restriction's
// gather of r at the tile's coarse faces
template <typename T, int DEG, int TW, int TH>
__device__ __forceinline__ void leg_down_body(const Blk& B, const LegArgs<T>& A, T* sm) {
  using G = DownTile<DEG, TW, TH>;
  constexpr int EW = G::EW;
  const Lvl& L = A.L;
  const Leg<T, G> g(L, (int)B.x * TW, (int)B.y * TH, sm);
  const int P = L.P, ov = (int)L.off[1], nx = g.nx, ny = g.ny;
  g.load_fold(A);
  // right-hand side: as given, or rU + G^T rD (restrict_flux2d_b_body)
  g.template over<0>([&](int, int i, int j) {
    Pair<T> z{(T)0, (T)0};
    if (g.inner || (i >= 0 && i <= nx && j >= 0 && j <= ny)) {
      const int id = j * P + i;
      z.u = GKB_LDG(A.b + id);
      z.v = GKB_LDG(A.b + ov + id);
      if (A.rd) {
        if (g.act_u(i, j)) z.u += slope_transpose<T, 0>(L, A.rd, i, j);
        if (g.act_v(i, j)) z.v += slope_transpose<T, 1>(L, A.rd, i, j);
      }
    }
    return z;
  }, [&](int o, const Pair<T>& z) {
    g.bu[o] = z.u;
    g.bv[o] = z.v;
  });
  __syncthreads();
  if (A.rd)
    g.template owned<TW, TH>(L, [&](int o, int id, int i, int j) {
      if (g.act_u(i, j)) A.bfull[id] = g.bu[o];
      if (g.act_v(i, j)) A.bfull[ov + id] = g.bv[o];
    });
  g.template cheb<1, true, true>(A, 0, g.bu, g.bv);
  if constexpr (DEG > 1) {
    g.template residual<2>(L);
    g.template cheb<3, false, false>(A, 1, g.ru, g.rv);
  }
  if constexpr (DEG > 2) {
    g.template residual<4>(L);
    g.template cheb<5, false, false>(A, 2, g.ru, g.rv);
  }
  g.template residual<2 * DEG>(L);
  g.template owned<TW, TH>(L, [&](int o, int id, int i, int j) {
    if (g.act_u(i, j)) A.xpre[id] = g.xu[o];
    if (g.act_v(i, j)) A.xpre[ov + id] = g.xv[o];
  });
  // gather at the coarse faces (restrict_flux_gather's terms and order)
  const Lvl& Lc = A.Lc;
  for (int t = g.tid; t < (TW / 2) * (TH / 2); t += LEG_NT) {
    const int J = t / (TW / 2), I = t - J * (TW / 2);
    const int gi = (int)B.x * (TW / 2) + I, gj = (int)B.y * (TH / 2) + J;
    if (gi >= Lc.n[0] || gj >= Lc.n[1]) continue;
    const int o = (G::HL + 2 * J) * EW + G::HL + 2 * I;  // the fine face (2I, 2J)
    const int id = gj * Lc.P + gi;
    T rU, rD;
    if (gi >= 1) {
      leg_gather<T>(g.ru, g.rv, o, 1, EW, rU, rD);
      A.bc[id] = rU;
      A.tmp[id] = rD;
    }
    if (gj >= 1) {
      leg_gather<T>(g.rv, g.ru, o, EW, 1, rU, rD);
      A.bc[(int)Lc.off[1] + id] = rU;
      A.tmp[(int)Lc.off[1] + id] = rD;
    }
  }
}

// x = xpre + P xc, then post-smoothing
template <typename T, int DEG, int TW, int TH>
__device__ __forceinline__ void leg_up_body(const Blk& B, const LegArgs<T>& A, T* sm) {
  using G = UpTile<DEG, TW, TH>;
  constexpr int EW = G::EW, EH = G::EH;
  const Lvl& L = A.L;
  const Lvl& Lc = A.Lc;
  const Leg<T, G> g(L, (int)B.x * TW, (int)B.y * TH, sm);
  const int P = L.P, ov = (int)L.off[1], nx = g.nx, ny = g.ny;
  g.load_fold(A);
  // the coarse correction of each coarse cell's 2 x 2 fine u and v faces
  // (prolong_flux2d_body), added once the iterate has been stored
  constexpr int CW = EW / 2, CN = CW * (EH / 2), CT = (CN + LEG_NT - 1) / LEG_NT;
  T e[CT][8];
#pragma unroll
  for (int k = 0; k < CT; ++k) {
    const int t = g.tid + k * LEG_NT;
    const int cj = t / CW;
    if (t < CN) leg_correction<T>(Lc, A.xc, g.ei / 2 + t - cj * CW, g.ej / 2 + cj, e[k]);
  }
  auto load = [&](const T* GKB_RESTRICT a, T* pu, T* pv) {
    g.template over<0>([&](int, int i, int j) {
      Pair<T> z{(T)0, (T)0};
      if (g.inner || (i >= 0 && i <= nx && j >= 0 && j <= ny)) {
        z.u = GKB_LDG(a + j * P + i);
        z.v = GKB_LDG(a + ov + j * P + i);
      }
      return z;
    }, [&](int o, const Pair<T>& z) {
      pu[o] = z.u;
      pv[o] = z.v;
    });
  };
  load(A.xpre, g.xu, g.xv);
  load(A.b, g.bu, g.bv);
  __syncthreads();
#pragma unroll
  for (int k = 0; k < CT; ++k) {
    const int t = g.tid + k * LEG_NT;
    if (t >= CN) break;
    const int cj = t / CW, o = 2 * cj * EW + 2 * (t - cj * CW);
    g.xu[o] += e[k][0];
    g.xu[o + EW] += e[k][1];
    g.xu[o + 1] += e[k][2];
    g.xu[o + EW + 1] += e[k][3];
    g.xv[o] += e[k][4];
    g.xv[o + 1] += e[k][5];
    g.xv[o + EW] += e[k][6];
    g.xv[o + EW + 1] += e[k][7];
  }
  __syncthreads();
  g.template residual<1>(L);
  g.template cheb<2, false, true>(A, 0, g.ru, g.rv);
  if constexpr (DEG > 1) {
    g.template residual<3>(L);
    g.template cheb<4, false, false>(A, 1, g.ru, g.rv);
  }
  if constexpr (DEG > 2) {
    g.template residual<5>(L);
    g.template cheb<6, false, false>(A, 2, g.ru, g.rv);
  }
  g.template owned<TW, TH>(L, [&](int o, int id, int i, int j) {
    if (g.act_u(i, j)) A.xout[id] = g.xu[o];
    if (g.act_v(i, j)) A.xout[ov + id] = g.xv[o];
  });
}

// ---------------------------------------------------------------------------
// The same legs for FP32 levels whose work is more than a few blocks: a thread
// keeps K consecutive rows of one column of the EW x EH tile (halo included)
// in registers (iterate, right-hand side, direction, residual) and reads only
// its neighbours from shared memory, so a smoothing step costs 14 shared
// accesses per position instead of 34 and no index arithmetic. All positions
// of the tile are computed in every step; what the halo has not reached is
// garbage that never enters the owned part.
// ---------------------------------------------------------------------------
template <int DEG, bool DOWN, int EW_, int EH_, int K_>
struct StripTile {
  static constexpr int EW = EW_, EH = EH_, K = K_, EN = EW * EH, NT = EN / K;
  static constexpr int HL = DOWN ? 2 * DEG + 2 : 2 * DEG, HH = 2 * DEG;
  static constexpr int TW = EW - HL - HH, TH = EH - HL - HH;  // owned cells
  static constexpr int PAD = EW + 32;                          // neighbours of the tile's rim read here
  static constexpr int PS = EN + PAD;
  // iterate and residual planes, then the class stencils (constant viscosity)
  // or the cell viscosities
  template <typename T>
  static constexpr size_t smem(bool var) { return (size_t)(4 * PS + PAD + (var ? PS : LEG_FOLD)) * sizeof(T); }
  static_assert(TW % 2 == 0 && TH % 2 == 0 && TW > 0 && TH > 0, "tiles own whole coarse cells");
};

template <typename T, class G, bool IN>
struct Strip {
  static constexpr int EW = G::EW, K = G::K;
  T *X0, *X1, *R0, *R1, *fold;   // planes of x and r (components 0, 1)
  int i, j, o, nx, ny, c, r0;    // this thread's column and first row: global, tile offset
  T xu[K], xv[K], bu[K], bv[K], du[K], dv[K], ru[K], rv[K];

  __device__ __forceinline__ Strip(const Lvl& L, int i0, int j0, T* sm) {
    X0 = sm + G::PAD;
    X1 = X0 + G::PS;
    R0 = X1 + G::PS;
    R1 = R0 + G::PS;
    fold = R1 + G::PS;
    c = threadIdx.x % EW;
    r0 = (int)(threadIdx.x / EW) * K;
    i = i0 - G::HL + c;
    j = j0 - G::HL + r0;
    o = r0 * EW + c;
    nx = L.n[0];
    ny = L.n[1];
  }
  __device__ __forceinline__ bool in_x() const { return i >= 0 && i < nx; }
  __device__ __forceinline__ bool act_u(int k) const { return IN || (i >= 1 && i < nx && j + k >= 0 && j + k < ny); }
  __device__ __forceinline__ bool act_v(int k) const { return IN || (i >= 0 && i < nx && j + k >= 1 && j + k < ny); }
  __device__ __forceinline__ void load(const T* GKB_RESTRICT a, int P, int ov, T* pu, T* pv) const {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const bool ok = IN || (i >= 0 && i <= nx && j + k >= 0 && j + k <= ny);
      const int id = (j + k) * P + i;
      pu[k] = ok ? GKB_LDG(a + id) : (T)0;
      pv[k] = ok ? GKB_LDG(a + ov + id) : (T)0;
    }
  }
  __device__ __forceinline__ void put(T* p0, T* p1, const T* a, const T* b) const {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      p0[o + k * EW] = a[k];
      p1[o + k * EW] = b[k];
    }
    __syncthreads();
  }

  // r = b - M x into the R planes
  __device__ __forceinline__ void residual(const Lvl& L) {
    const bool gd = L.has_gd;
    T cu[K + 2], cv[K + 2], rr[K + 1], lv[K + 1];  // cu, cv: rows -1 .. K; rr: u right of rows -1 .. K-1; lv: rows 0 .. K
    cu[0] = X0[o - EW];
    cv[0] = X1[o - EW];
    cu[K + 1] = X0[o + K * EW];
    cv[K + 1] = X1[o + K * EW];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      cu[k + 1] = xu[k];
      cv[k + 1] = xv[k];
    }
#pragma unroll
    for (int k = 0; k <= K; ++k) {
      rr[k] = X0[o + (k - 1) * EW + 1];
      lv[k] = X1[o + k * EW - 1];
    }
    T dlo = cu[0] - rr[0] + cv[0] - cv[1];  // divergence of the cell below row 0
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const T lu = X0[o + k * EW - 1], rw = X1[o + k * EW + 1];
      const T d0 = cu[k + 1] - rr[k + 1] + cv[k + 1] - cv[k + 2];
      const T dl = lu - cu[k + 1] + lv[k] - lv[k + 1];
      const T au = rr[k + 1] + lu + cu[k + 2] + cu[k];
      const T av = rw + lv[k] + cv[k + 2] + cv[k];
      T zu = const_row<T, 0>(L, bu[k], cu[k + 1], au, gd, d0, dl);
      T zv = const_row<T, 0>(L, bv[k], cv[k + 1], av, gd, d0, dlo);
      if (!IN) {
        const int jj = j + k;
        const T g2 = Kc<T>::g2(L), mu = Kc<T>::mu0(L), ws = Kc<T>::ws(L);
        // faces beside a wall of their tangential axis (w_row's links)
        if (jj == 0 || jj == ny - 1) {
          T w = fma(mu, cu[k + 1] - rr[k + 1], (T)0);
          w = fma(mu, cu[k + 1] - lu, w);
          w = jj == ny - 1 ? fma((T)2 * mu, cu[k + 1], w) : fma(mu, cu[k + 1] - cu[k + 2], w);
          w = jj == 0 ? fma((T)2 * mu, cu[k + 1], w) : fma(mu, cu[k + 1] - cu[k], w);
          zu = bu[k] - wall_row<T>(w, ws, gd, g2, d0, dl);
        }
        if (i == 0 || i == nx - 1) {
          T w = fma(mu, cv[k + 1] - cv[k + 2], (T)0);
          w = fma(mu, cv[k + 1] - cv[k], w);
          w = i == nx - 1 ? fma((T)2 * mu, cv[k + 1], w) : fma(mu, cv[k + 1] - rw, w);
          w = i == 0 ? fma((T)2 * mu, cv[k + 1], w) : fma(mu, cv[k + 1] - lv[k], w);
          zv = bv[k] - wall_row<T>(w, ws, gd, g2, d0, dlo);
        }
        if (!act_u(k)) zu = (T)0;
        if (!act_v(k)) zv = (T)0;
      }
      ru[k] = zu;
      rv[k] = zv;
      dlo = d0;
    }
    put(R0, R1, ru, rv);
  }

  // one Chebyshev step from the source in the R planes (own rows: su, sv)
  template <bool ZERO, bool FIRST>
  __device__ __forceinline__ void cheb(const LegArgs<T>& A, int s, const T* su, const T* sv) {
    const T ca = A.ca[s], cb = A.cb[s];
    T cu[K + 2], cv[K + 1], rr[K + 1], lv[K + 1];
    cu[0] = R0[o - EW];
    cu[K + 1] = R0[o + K * EW];
    cv[K] = R1[o + K * EW];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      cu[k + 1] = su[k];
      cv[k] = sv[k];
    }
#pragma unroll
    for (int k = 0; k <= K; ++k) {
      rr[k] = R0[o + (k - 1) * EW + 1];
      lv[k] = R1[o + k * EW - 1];
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const T rw = R1[o + k * EW + 1];
      const T qu[7] = {cu[k + 1], cu[k], lv[k], cv[k], cu[k + 2], lv[k + 1], cv[k + 1]};
      const T qv[7] = {cv[k], cu[k], cu[k + 1], lv[k], rr[k], rr[k + 1], rw};
      T zu, zv;
      if (IN) {
        zu = mul_rn(A.fs[s].c[0][0], qu[0]);
        zv = mul_rn(A.fs[s].c[1][0], qv[0]);
#pragma unroll
        for (int q = 1; q < 7; ++q) {
          zu = fma(A.fs[s].c[0][q], qu[q], zu);
          zv = fma(A.fs[s].c[1][q], qv[q], zv);
        }
        if (!FIRST) {
          zu = fma(cb, du[k], zu);
          zv = fma(cb, dv[k], zv);
        }
      } else {
        const int jj = j + k;
        zu = zv = (T)0;
        if (in_x() && jj >= 0 && jj < ny) {
          const bool sc = cheb2_scaled(A.L, i, jj);
          const T* f = fold + (sc ? FOLD2_CLASSES + s : cls7(i, nx) * 7 + cls7(jj, ny)) * 14;
          T wu = mul_rn(f[0], qu[0]), wv = mul_rn(f[7], qv[0]);
#pragma unroll
          for (int q = 1; q < 7; ++q) {
            wu = fma(f[q], qu[q], wu);
            wv = fma(f[7 + q], qv[q], wv);
          }
          if (i >= 1) zu = cheb_wall<T>(sc ? (T)1 : ca, wu, cb, FIRST ? (T)0 : du[k], FIRST);
          if (jj >= 1) zv = cheb_wall<T>(sc ? (T)1 : ca, wv, cb, FIRST ? (T)0 : dv[k], FIRST);
        }
      }
      du[k] = zu;
      dv[k] = zv;
      xu[k] = ZERO ? zu : xu[k] + zu;
      xv[k] = ZERO ? zv : xv[k] + zv;
    }
    put(X0, X1, xu, xv);
  }

  // write the owned rows of (a, b)
  __device__ __forceinline__ void store(T* GKB_RESTRICT y, int P, int ov, const T* a, const T* b) const {
    if (c < G::HL || c >= G::HL + G::TW) return;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      if (r0 + k < G::HL || r0 + k >= G::HL + G::TH) continue;
      const int id = (j + k) * P + i;
      if (act_u(k)) y[id] = a[k];
      if (act_v(k)) y[ov + id] = b[k];
    }
  }
  __device__ __forceinline__ void setup(const LegArgs<T>& A) const {
    for (int t = IN ? LEG_FOLD : (int)threadIdx.x; t < LEG_FOLD; t += G::NT) fold[t] = leg_fold_entry(A, t);
  }
};

// Variable viscosity: the plane after the residual holds the cells' viscosity
// (0 outside the domain), from which every link forms its node mean; the
// smoother reads the patch inverses (10 planes of A.table) once per step, and
// the tile's 40 bytes per node stay in L1 between the steps. The operations
// are those of the general variable-viscosity row (w_row) and of k_cheb.
template <typename T, class G, bool IN>
struct StripVar : Strip<T, G, IN> {
  using S = Strip<T, G, IN>;
  using S::X0; using S::X1; using S::R0; using S::R1; using S::i; using S::j; using S::o; using S::nx; using S::ny;
  using S::xu; using S::xv; using S::bu; using S::bv; using S::du; using S::dv; using S::ru; using S::rv;
  static constexpr int EW = G::EW, K = G::K;
  T* MU;
  __device__ __forceinline__ StripVar(const Lvl& L, int i0, int j0, T* sm) : S(L, i0, j0, sm) { MU = S::fold; }
  __device__ __forceinline__ void setup(const LegArgs<T>& A) const {
    const T* mu = MuPtr<T>::get(A.L);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const bool ok = IN || (i >= 0 && i < nx && j + k >= 0 && j + k < ny);
      MU[o + k * EW] = ok ? GKB_LDG(mu + (j + k) * A.L.P + i) : (T)0;
    }
  }

  __device__ __forceinline__ void residual(const Lvl& L) {
    const bool gd = L.has_gd;
    const T g2 = Kc<T>::g2(L), ws = Kc<T>::ws(L);
    T cu[K + 2], cv[K + 2], rr[K + 1], lv[K + 1];  // as in Strip
    T cm[K + 2], lm[K + 2];                        // viscosity of rows -1 .. K, own column and the one left of it
    cu[0] = X0[o - EW];
    cv[0] = X1[o - EW];
    cu[K + 1] = X0[o + K * EW];
    cv[K + 1] = X1[o + K * EW];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      cu[k + 1] = xu[k];
      cv[k + 1] = xv[k];
    }
#pragma unroll
    for (int k = 0; k <= K; ++k) {
      rr[k] = X0[o + (k - 1) * EW + 1];
      lv[k] = X1[o + k * EW - 1];
    }
#pragma unroll
    for (int k = 0; k < K + 2; ++k) {
      cm[k] = MU[o + (k - 1) * EW];
      lm[k] = MU[o + (k - 1) * EW - 1];
    }
    // node means as edge_mu_cells sums them, per component: over the cells at
    // (C-1, A-1), (C-1, A), (C, A-1), (C, A)
    auto mean_u = [&](int k) -> T {  // node (i, j + k)
      const T s = ((lm[k] + lm[k + 1]) + cm[k]) + cm[k + 1];
      return s * ((!IN && (j + k == 0 || j + k == ny)) ? (T)0.5 : (T)0.25);
    };
    T mu_lo = mean_u(0);
    T rm_lo = MU[o - EW + 1];
    T dlo = cu[0] - rr[0] + cv[0] - cv[1];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const T lu = X0[o + k * EW - 1], rw = X1[o + k * EW + 1], rm = MU[o + k * EW + 1];
      const T d0 = cu[k + 1] - rr[k + 1] + cv[k + 1] - cv[k + 2];
      const T dl = lu - cu[k + 1] + lv[k] - lv[k + 1];
      const T m0 = cm[k + 1], xf = cu[k + 1], yf = cv[k + 1];
      const T mu_hi = mean_u(k + 1);
      const T sl = ((lm[k] + cm[k]) + lm[k + 1]) + cm[k + 1];   // node (i, j + k), v's order
      const T sr = ((cm[k] + rm_lo) + cm[k + 1]) + rm;          // node (i + 1, j + k)
      T mv_lo = sl * (T)0.25, mv_hi = sr * (T)0.25;
      if (!IN) {
        if (i == 0) mv_lo = sl * (T)0.5;
        if (i == nx - 1) mv_hi = sr * (T)0.5;
      }
      T w = fma(m0, xf - rr[k + 1], (T)0);
      w = fma(lm[k + 1], xf - lu, w);
      if (IN) {
        w = fma(mu_hi, xf - cu[k + 2], w);
        w = fma(mu_lo, xf - cu[k], w);
      } else {
        w = j + k == ny - 1 ? fma((T)2 * mu_hi, xf, w) : fma(mu_hi, xf - cu[k + 2], w);
        w = j + k == 0 ? fma((T)2 * mu_lo, xf, w) : fma(mu_lo, xf - cu[k], w);
      }
      T y = fma(m0, yf - cv[k + 2], (T)0);
      y = fma(cm[k], yf - cv[k], y);
      if (IN) {
        y = fma(mv_hi, yf - rw, y);
        y = fma(mv_lo, yf - lv[k], y);
      } else {
        y = i == nx - 1 ? fma((T)2 * mv_hi, yf, y) : fma(mv_hi, yf - rw, y);
        y = i == 0 ? fma((T)2 * mv_lo, yf, y) : fma(mv_lo, yf - lv[k], y);
      }
      const T zu = bu[k] - wall_row<T>(w, ws, gd, g2, d0, dl);
      const T zv = bv[k] - wall_row<T>(y, ws, gd, g2, d0, dlo);
      ru[k] = this->act_u(k) ? zu : (T)0;
      rv[k] = this->act_v(k) ? zv : (T)0;
      dlo = d0;
      mu_lo = mu_hi;
      rm_lo = rm;
    }
    this->put(R0, R1, ru, rv);
  }

  template <bool ZERO, bool FIRST>
  __device__ __forceinline__ void cheb(const LegArgs<T>& A, int s, const T* su, const T* sv) {
    const T ca = A.ca[s], cb = A.cb[s];
    const long long Q = vtab_plane(A.L);
    const int P = A.L.P;
    T cu[K + 2], cv[K + 1], rr[K + 1], lv[K + 1];
    cu[0] = R0[o - EW];
    cu[K + 1] = R0[o + K * EW];
    cv[K] = R1[o + K * EW];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      cu[k + 1] = su[k];
      cv[k] = sv[k];
    }
#pragma unroll
    for (int k = 0; k <= K; ++k) {
      rr[k] = R0[o + (k - 1) * EW + 1];
      lv[k] = R1[o + k * EW - 1];
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
      T zu = (T)0, zv = (T)0;
      if (IN || (this->in_x() && j + k >= 0 && j + k < ny)) {
        const T rw = R1[o + k * EW + 1];
        const T* t = A.table + (j + k) * P + i;
        auto at = [&](const T* q, int r, int c) { return GKB_LDG(q + sym4(r, c) * Q); };
        // the patches of the nodes (i, j), (i, j + 1) and (i + 1, j)
        const T t13 = at(t, 1, 3);
        const T a1 = patch_dot<T>(at(t, 1, 0), at(t, 1, 1), at(t, 1, 2), t13, cu[k], cu[k + 1], lv[k], cv[k]);
        const T a3 = patch_dot<T>(at(t, 3, 0), t13, at(t, 3, 2), at(t, 3, 3), cu[k], cu[k + 1], lv[k], cv[k]);
        const T a0 = patch_dot<T>(at(t + P, 0, 0), at(t + P, 0, 1), at(t + P, 0, 2), at(t + P, 0, 3), cu[k + 1],
                                  cu[k + 2], lv[k + 1], cv[k + 1]);
        const T a2 = patch_dot<T>(at(t + 1, 2, 0), at(t + 1, 2, 1), at(t + 1, 2, 2), at(t + 1, 2, 3), rr[k], rr[k + 1],
                                  cv[k], rw);
        if (this->act_u(k)) zu = cheb_wall<T>(ca, a1 + a0, cb, FIRST ? (T)0 : du[k], FIRST);
        if (this->act_v(k)) zv = cheb_wall<T>(ca, a3 + a2, cb, FIRST ? (T)0 : dv[k], FIRST);
      }
      du[k] = zu;
      dv[k] = zv;
      xu[k] = ZERO ? zu : xu[k] + zu;
      xv[k] = ZERO ? zv : xv[k] + zv;
    }
    this->put(X0, X1, xu, xv);
  }
};

// the tile's place: every position whose row or stencil is formed is interior
template <class G>
__device__ __forceinline__ bool strip_inner(const Blk& B, const Lvl& L) {
  const int ei = (int)B.x * G::TW - G::HL, ej = (int)B.y * G::TH - G::HL;
  return leg_inner(L, ei, ei + G::EW - 1, ej, ej + G::EH - 1);
}

template <typename T, int DEG, class G, class S>
__device__ __forceinline__ void strip_down_in(const Blk& B, const LegArgs<T>& A, T* sm) {
  constexpr int EW = G::EW, K = G::K;
  const Lvl& L = A.L;
  const int P = L.P, ov = (int)L.off[1];
  S g(L, (int)B.x * G::TW, (int)B.y * G::TH, sm);
  g.setup(A);
  g.load(A.b, P, ov, g.bu, g.bv);
  if (A.rd) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      if (g.act_u(k)) g.bu[k] += slope_transpose<T, 0>(L, A.rd, g.i, g.j + k);
      if (g.act_v(k)) g.bv[k] += slope_transpose<T, 1>(L, A.rd, g.i, g.j + k);
    }
    g.store(A.bfull, P, ov, g.bu, g.bv);
  }
  g.put(g.R0, g.R1, g.bu, g.bv);
  g.template cheb<true, true>(A, 0, g.bu, g.bv);
  if constexpr (DEG > 1) {
    g.residual(L);
    g.template cheb<false, false>(A, 1, g.ru, g.rv);
  }
  if constexpr (DEG > 2) {
    g.residual(L);
    g.template cheb<false, false>(A, 2, g.ru, g.rv);
  }
  g.store(A.xpre, P, ov, g.xu, g.xv);
  g.residual(L);
  const Lvl& Lc = A.Lc;
  constexpr int CW = G::TW / 2, CN = CW * (G::TH / 2);
  for (int t = threadIdx.x; t < CN; t += G::NT) {
    const int J = t / CW, I = t - J * CW;
    const int gi = (int)B.x * CW + I, gj = (int)B.y * (G::TH / 2) + J;
    if (gi >= Lc.n[0] || gj >= Lc.n[1]) continue;
    const int o = (G::HL + 2 * J) * EW + G::HL + 2 * I;
    const int id = gj * Lc.P + gi;
    T rU, rD;
    if (gi >= 1) {
      leg_gather<T>(g.R0, g.R1, o, 1, EW, rU, rD);
      A.bc[id] = rU;
      A.tmp[id] = rD;
    }
    if (gj >= 1) {
      leg_gather<T>(g.R1, g.R0, o, EW, 1, rU, rD);
      A.bc[(int)Lc.off[1] + id] = rU;
      A.tmp[(int)Lc.off[1] + id] = rD;
    }
  }
}

template <typename T, int DEG, class G, class S>
__device__ __forceinline__ void strip_up_in(const Blk& B, const LegArgs<T>& A, T* sm) {
  constexpr int EW = G::EW, K = G::K;
  const Lvl& L = A.L;
  const int P = L.P, ov = (int)L.off[1];
  S g(L, (int)B.x * G::TW, (int)B.y * G::TH, sm);
  g.setup(A);
  g.load(A.xpre, P, ov, g.xu, g.xv);
  g.load(A.b, P, ov, g.bu, g.bv);
  g.put(g.X0, g.X1, g.xu, g.xv);
  constexpr int CW = EW / 2, CN = CW * (G::EH / 2);
  const int ci0 = ((int)B.x * G::TW - G::HL) / 2, cj0 = ((int)B.y * G::TH - G::HL) / 2;
  for (int t = threadIdx.x; t < CN; t += G::NT) {
    const int cj = t / CW, ci = t - cj * CW;
    T e[8];
    leg_correction<T>(A.Lc, A.xc, ci0 + ci, cj0 + cj, e);
    const int o = 2 * cj * EW + 2 * ci;
    g.X0[o] += e[0];
    g.X0[o + EW] += e[1];
    g.X0[o + 1] += e[2];
    g.X0[o + EW + 1] += e[3];
    g.X1[o] += e[4];
    g.X1[o + 1] += e[5];
    g.X1[o + EW] += e[6];
    g.X1[o + EW + 1] += e[7];
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < K; ++k) {
    g.xu[k] = g.X0[g.o + k * EW];
    g.xv[k] = g.X1[g.o + k * EW];
  }
  g.residual(L);
  g.template cheb<false, true>(A, 0, g.ru, g.rv);
  if constexpr (DEG > 1) {
    g.residual(L);
    g.template cheb<false, false>(A, 1, g.ru, g.rv);
  }
  if constexpr (DEG > 2) {
    g.residual(L);
    g.template cheb<false, false>(A, 2, g.ru, g.rv);
  }
  g.store(A.xout, P, ov, g.xu, g.xv);
}

template <typename T, int DEG, class G, bool DOWN, template <typename, class, bool> class S>
__device__ __forceinline__ void strip_body(const Blk& B, const LegArgs<T>& A, T* sm) {
  const bool in = strip_inner<G>(B, A.L);
  if constexpr (DOWN) {
    if (in) strip_down_in<T, DEG, G, S<T, G, true>>(B, A, sm);
    else strip_down_in<T, DEG, G, S<T, G, false>>(B, A, sm);
  } else {
    if (in) strip_up_in<T, DEG, G, S<T, G, true>>(B, A, sm);
    else strip_up_in<T, DEG, G, S<T, G, false>>(B, A, sm);
  }
}

// how a level's legs are tiled; LEG_OFF: separate launches
enum LegKind { LEG_OFF = 0, LEG_8, LEG_STRIP, LEG_VAR };

// geometry and body of one leg of kind KIND
template <int DEG, int KIND, bool DOWN>
struct LegShape {
  static constexpr int TILE = 8;
  using G = std::conditional_t<DOWN, DownTile<DEG, TILE, TILE>, UpTile<DEG, TILE, TILE>>;
  static constexpr int NT = LEG_NT, TW = TILE, TH = TILE;
  template <typename T>
  static constexpr size_t smem() { return leg_smem<T, G>(); }
  static dim3 grid(const Lvl& L) { return dim3((L.n[0] + TW - 1) / TW, (L.n[1] + TH - 1) / TH, 1); }
};
template <class G_, bool VAR>
struct StripShape {
  using G = G_;
  static constexpr int NT = G::NT, TW = G::TW, TH = G::TH;
  template <typename T>
  static constexpr size_t smem() { return G::template smem<T>(VAR); }
  static dim3 grid(const Lvl& L) { return dim3((L.n[0] + TW - 1) / TW, (L.n[1] + TH - 1) / TH, 1); }
};
// 1024^2 mixed solves by tile: constant viscosity 64 x 32 61.8 ms, 32 x 32
// 62.4, 64 x 64 77.0; variable 32 x 32 at two blocks per SM (128 registers)
// 104 ms, at three (80) 108, 64 x 32 109. Eight rows per thread instead of
// four: 69 ms (half the warps in flight).
template <int DEG, bool DOWN>
struct LegShape<DEG, LEG_STRIP, DOWN> : StripShape<StripTile<DEG, DOWN, 64, 32, 4>, false> {};
template <int DEG, bool DOWN>
struct LegShape<DEG, LEG_VAR, DOWN> : StripShape<StripTile<DEG, DOWN, 32, 32, 4>, true> {};

template <typename T, int DEG, int KIND, bool DOWN>
__device__ __forceinline__ void leg_body(const Blk& B, const LegArgs<T>& A, T* sm) {
  using S = LegShape<DEG, KIND, DOWN>;
  if constexpr (KIND == LEG_STRIP) strip_body<T, DEG, typename S::G, DOWN, Strip>(B, A, sm);
  else if constexpr (KIND == LEG_VAR) strip_body<T, DEG, typename S::G, DOWN, StripVar>(B, A, sm);
  else if constexpr (DOWN) leg_down_body<T, DEG, S::TILE, S::TILE>(B, A, sm);
  else leg_up_body<T, DEG, S::TILE, S::TILE>(B, A, sm);
}

}  // namespace gkb
