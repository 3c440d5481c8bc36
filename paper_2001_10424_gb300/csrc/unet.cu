// unet.cu - U-Net kernels (forward FP32 and BF16 tensor cores, backward,
// Adam) and the gkb_unet_* entry points.
//
// Layout: activations NHWC FP32; parameters flat FP32, per layer the weights
// w[ky][kx][cin][cout] then the bias. A convolution input can be the channel
// concatenation of two tensors, the first one read at half resolution with
// bilinear doubling folded into the fetch (pixel-centre alignment: fine pixel
// 2k takes 3/4 of coarse k and 1/4 of k - 1, fine 2k + 1 takes 3/4 of k and
// 1/4 of k + 1, neighbours clamped at the edge).
#include <cuda_bf16.h>
#include <math.h>

#include <cmath>

#include <algorithm>
#include <new>
#include <random>
#include <string>
#include <vector>

#include "../../include/gkb.h"
#include "prof.h"
#include "unet.cuh"

namespace gkb {

struct In2 {
  const float* p0;  // first input (channels [0, c0))
  int c0;
  int up0;          // 1: p0 has half the resolution (nearest upsampling)
  const float* p1;  // second input (channels [c0, c0 + c1)), full resolution
  int c1;
  int v4;           // 1: groups of four channels may be read as one vector
};

// an input of the network; a caller's image need not be 16-byte aligned
static In2 make_in(const float* p0, int c0, int up0 = 0, const float* p1 = nullptr, int c1 = 0) {
  const bool v4 = c0 % 4 == 0 && c1 % 4 == 0 && ((uintptr_t)p0 & 15) == 0 && ((uintptr_t)p1 & 15) == 0;
  return In2{p0, c0, up0, p1, c1, v4 ? 1 : 0};
}

constexpr int UT = 256;  // threads per block of the FP32 kernels

// coarse row (or column) pair of a fine index under bilinear doubling
__device__ __forceinline__ void up_pair(int f, int m, int& k, int& k2) {
  k = f >> 1;
  k2 = (f & 1) ? min(k + 1, m - 1) : max(k - 1, 0);
}

// 3/4 x 3/4, 3/4 x 1/4, 1/4 x 3/4 and 1/4 x 1/4 of the four coarse values
__device__ __forceinline__ float bilin(float a, float b, float c, float d) {
  return fmaf(0.0625f, d, fmaf(0.1875f, c, fmaf(0.1875f, b, 0.5625f * a)));
}

// channel ci of the (concatenated) input at full-resolution pixel (yy, xx)
__device__ __forceinline__ float in_val(const In2& in, int b, int yy, int xx, int h, int wd, int ci) {
  if (ci < in.c0) {
    if (!in.up0) return __ldg(in.p0 + (((long long)b * h + yy) * wd + xx) * in.c0 + ci);
    const int h0 = h >> 1, w0 = wd >> 1;
    int k, k2, l, l2;
    up_pair(yy, h0, k, k2);
    up_pair(xx, w0, l, l2);
    const float* base = in.p0 + (long long)b * h0 * w0 * in.c0 + ci;
    return bilin(__ldg(base + ((long long)k * w0 + l) * in.c0), __ldg(base + ((long long)k * w0 + l2) * in.c0),
                 __ldg(base + ((long long)k2 * w0 + l) * in.c0), __ldg(base + ((long long)k2 * w0 + l2) * in.c0));
  }
  return __ldg(in.p1 + (((long long)b * h + yy) * wd + xx) * in.c1 + (ci - in.c0));
}

__device__ __forceinline__ void px_decode(long long p, int h, int w, int& b, int& y, int& x) {
  x = (int)(p % w);
  const long long q = p / w;
  y = (int)(q % h);
  b = (int)(q / h);
}

// four consecutive channels [ci, ci + 4), ci < cin a multiple of 4, of the
// (concatenated) input at full-resolution pixel (yy, xx), zero past cin
__device__ __forceinline__ float4 in_val4(const In2& in, int b, int yy, int xx, int h, int wd, int ci, int cin) {
  if (in.v4) {
    if (ci < in.c0) {
      if (!in.up0)
        return __ldg(reinterpret_cast<const float4*>(in.p0 + (((long long)b * h + yy) * wd + xx) * in.c0 + ci));
      const int h0 = h >> 1, w0 = wd >> 1;
      int k, k2, l, l2;
      up_pair(yy, h0, k, k2);
      up_pair(xx, w0, l, l2);
      const float* base = in.p0 + (long long)b * h0 * w0 * in.c0 + ci;
      auto at = [&](int kk, int ll) {
        return __ldg(reinterpret_cast<const float4*>(base + ((long long)kk * w0 + ll) * in.c0));
      };
      const float4 p = at(k, l), q = at(k, l2), r = at(k2, l), s = at(k2, l2);
      return make_float4(bilin(p.x, q.x, r.x, s.x), bilin(p.y, q.y, r.y, s.y), bilin(p.z, q.z, r.z, s.z),
                         bilin(p.w, q.w, r.w, s.w));
    }
    return __ldg(reinterpret_cast<const float4*>(in.p1 + (((long long)b * h + yy) * wd + xx) * in.c1 + (ci - in.c0)));
  }
  float4 v;
  v.x = ci + 0 < cin ? in_val(in, b, yy, xx, h, wd, ci + 0) : 0.f;
  v.y = ci + 1 < cin ? in_val(in, b, yy, xx, h, wd, ci + 1) : 0.f;
  v.z = ci + 2 < cin ? in_val(in, b, yy, xx, h, wd, ci + 2) : 0.f;
  v.w = ci + 3 < cin ? in_val(in, b, yy, xx, h, wd, ci + 3) : 0.f;
  return v;
}

// ---------------------------------------------------------------------------
// FP32 3x3 convolutions: forward, and the data gradient (the same convolution
// with the taps mirrored and the weights transposed). Bound by the FP32 pipe
// once their operands come from shared memory and registers: a thread forms
// CVR rows x COT outputs of one pixel column, so every staged input and every
// (broadcast) weight it reads serves COT or CVR multiply-adds; one thread per
// pixel read a weight per multiply-add. Block: 32 columns x (CVR RG) rows of
// pixels, CG groups of COT outputs; inputs staged as channel planes with a
// one-pixel halo. Measured on 8 images of 512^2 (FP32 peak 72 TFLOP/s): 16 ->
// 16 forward 0.28 ms (35 TFLOP/s), the concatenated 48 -> 16 with its bilinear
// input 1.29 ms (22), its data gradient 0.73-0.85 ms (34-40); forward and data
// gradient together were 11.3 and about 15 ms.
// ---------------------------------------------------------------------------
constexpr int CVK = 8;       // input channels per chunk
constexpr int CVR = 4;       // rows per thread
constexpr int CVP = 36;      // row pitch of a staged plane

struct ConvArgs {
  In2 in;
  const float* w;     // weights, [tap][ci][co] of the forward layer
  const float* bias;
  float* o0;          // output channels [0, oc0)
  float* o1;          // and the rest
  const float* m0;    // with m0: outputs of o0 are zeroed where m0 is not positive
  int oc0, cin, cout, relu, n, h, wd;
};

// plane stride 12 mod 32 words: the four channels of a staged pixel and its
// neighbour's land in distinct banks
template <int RG>
struct ConvSmem {
  static constexpr int rows = CVR * RG + 2;
  static constexpr int plane = (rows * CVP + 31) / 32 * 32 + 12;
};

// 8 floats as one 32-byte store
__device__ __forceinline__ void st8(float* p, const float* v) {
  asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]),
               "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
               : "memory");
}

// put(k, v): item k = tid, tid + nt, ... < items of a staged tile, v = load(k);
// U loads are issued before the first is stored (one at a time, staging a
// 48-channel tile took longer than its multiply-adds)
template <int U, class Load, class Put>
__device__ __forceinline__ void stage(int items, int nt, Load load, Put put) {
  for (int t0 = threadIdx.x; t0 < items; t0 += U * nt) {
    float4 v[U];
#pragma unroll
    for (int k = 0; k < U; ++k)
      if (t0 + k * nt < items) v[k] = load(t0 + k * nt);
#pragma unroll
    for (int k = 0; k < U; ++k)
      if (t0 + k * nt < items) put(t0 + k * nt, v[k]);
  }
}

// channels [c0, c0 + nc) (nc a multiple of 4) of the block's tile into planes
template <int RG>
__device__ __forceinline__ void stage_planes(const ConvArgs& A, float* xs, int b, int x0, int y0, int c0, int nc, int nt) {
  using SM = ConvSmem<RG>;
  const int ng = nc / 4;
  stage<4>(SM::rows * 34 * ng, nt, [&](int t) {
    const int g = t % ng, px = t / ng, r = px / 34;
    const int yy = y0 + r - 1, xx = x0 + px - r * 34 - 1, ci = c0 + 4 * g;
    if (yy >= 0 && yy < A.h && xx >= 0 && xx < A.wd && ci < A.cin) return in_val4(A.in, b, yy, xx, A.h, A.wd, ci, A.cin);
    return make_float4(0.f, 0.f, 0.f, 0.f);
  }, [&](int t, const float4& v) {
    const int g = t % ng, px = t / ng, r = px / 34;
    float* d = xs + 4 * g * SM::plane + r * CVP + px - r * 34;
    d[0] = v.x;
    d[SM::plane] = v.y;
    d[2 * SM::plane] = v.z;
    d[3 * SM::plane] = v.w;
  });
}

// COT weights at wp, COT x CVR multiply-adds
template <int COT>
__device__ __forceinline__ void conv_fma(float (&acc)[CVR][COT], const float (&v)[CVR], const float* wp) {
  float wv[COT];
#pragma unroll
  for (int o = 0; o < COT; o += 4) {
    const float4 q = *reinterpret_cast<const float4*>(wp + o);
    wv[o] = q.x;
    wv[o + 1] = q.y;
    wv[o + 2] = q.z;
    wv[o + 3] = q.w;
  }
#pragma unroll
  for (int r = 0; r < CVR; ++r)
#pragma unroll
    for (int o = 0; o < COT; ++o) acc[r][o] = fmaf(v[r], wv[o], acc[r][o]);
}

// write a thread's CVR x COT outputs
template <int COT>
__device__ __forceinline__ void conv_store(const ConvArgs& A, float (&acc)[CVR][COT], int b, int x, int y0, int cb) {
  if (x >= A.wd) return;
  const bool first = cb < A.oc0;  // a group's outputs lie in one of the two arrays
  float* out = first ? A.o0 : A.o1;
  const int oc = first ? A.oc0 : A.cout - A.oc0, ob = first ? cb : cb - A.oc0;
#pragma unroll
  for (int r = 0; r < CVR; ++r) {
    if (y0 + r >= A.h) break;
    const long long at = (((long long)b * A.h + y0 + r) * A.wd + x) * oc + ob;
    if (A.relu)
#pragma unroll
      for (int o = 0; o < COT; ++o) acc[r][o] = fmaxf(acc[r][o], 0.f);
    if (A.m0 && first) {
#pragma unroll
      for (int o = 0; o < COT; o += 4) {
        const float4 m = __ldg(reinterpret_cast<const float4*>(A.m0 + at + o));
        if (!(m.x > 0.f)) acc[r][o] = 0.f;
        if (!(m.y > 0.f)) acc[r][o + 1] = 0.f;
        if (!(m.z > 0.f)) acc[r][o + 2] = 0.f;
        if (!(m.w > 0.f)) acc[r][o + 3] = 0.f;
      }
    }
    if constexpr (COT % 8 == 0) {
#pragma unroll
      for (int o = 0; o < COT; o += 8) st8(out + at + o, &acc[r][o]);
    } else {
#pragma unroll
      for (int o = 0; o < COT; ++o)
        if (cb + o < A.cout) out[at + o] = acc[r][o];
    }
  }
}

// Forward. Every output is the chain bias, then tap by tap, within a tap
// channel by channel: the order does not depend on the tiling, so neither do
// the signs the ReLUs see (one activation in 1e8 lies within rounding of zero,
// and where its sign flips the gradient moves by more than all other rounding
// of a training step). So all channels and weights are staged at once.
template <int COT, int CG, int RG>
__global__ void __launch_bounds__(32 * CG * RG) k_conv_fwd(const ConvArgs A) {
  using SM = ConvSmem<RG>;
  constexpr int CO = COT * CG, NT = 32 * CG * RG;
  extern __shared__ __align__(16) float cv_sm[];
  const int nc = (A.cin + 3) / 4 * 4;
  float* xs = cv_sm;
  float* ws = cv_sm + nc * SM::plane;  // [tap][ci][CO]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rg = warp % RG, cg = warp / RG;
  const int x0 = blockIdx.x * 32, y0 = blockIdx.y * (CVR * RG);
  for (int t = tid; t < 9 * A.cin * CO; t += NT) {
    const int o = t % CO;
    ws[t] = o < A.cout ? __ldg(A.w + (t / CO) * A.cout + o) : 0.f;
  }
  for (int b = blockIdx.z; b < A.n; b += gridDim.z) {
    float acc[CVR][COT];
#pragma unroll
    for (int o = 0; o < COT; ++o) {
      const int co = cg * COT + o;
      const float v = co < A.cout ? __ldg(A.bias + co) : 0.f;
#pragma unroll
      for (int r = 0; r < CVR; ++r) acc[r][o] = v;
    }
    __syncthreads();  // the previous image's reads
    stage_planes<RG>(A, xs, b, x0, y0, 0, nc, NT);
    __syncthreads();
    const float* wp = ws + cg * COT;
#pragma unroll 1
    for (int tap = 0; tap < 9; ++tap) {
      const float* xp = xs + (rg * CVR + tap / 3) * CVP + lane + tap % 3;
#pragma unroll 4
      for (int ci = 0; ci < A.cin; ++ci) {
        float v[CVR];
#pragma unroll
        for (int r = 0; r < CVR; ++r) v[r] = xp[ci * SM::plane + r * CVP];
        conv_fma<COT>(acc, v, wp);
        wp += CO;
      }
    }
    conv_store<COT>(A, acc, b, x0 + lane, y0 + rg * CVR, cg * COT);
  }
}

// Data gradient, the channels in chunks of CVK: per channel a thread keeps the
// 18 inputs of its rows in registers for all nine taps.
template <int COT, int CG, int RG>
__global__ void __launch_bounds__(32 * CG * RG, CG * RG <= 8 ? 2 : 1) k_conv_bwd(const ConvArgs A) {
  using SM = ConvSmem<RG>;
  constexpr int CO = COT * CG, NT = 32 * CG * RG;
  __shared__ __align__(16) float xs[CVK * SM::plane];
  __shared__ __align__(16) float ws[CVK * 9 * CO];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rg = warp % RG, cg = warp / RG;
  const int x0 = blockIdx.x * 32, y0 = blockIdx.y * (CVR * RG);
  for (int b = blockIdx.z; b < A.n; b += gridDim.z) {
    float acc[CVR][COT];
#pragma unroll
    for (int o = 0; o < COT; ++o)
#pragma unroll
      for (int r = 0; r < CVR; ++r) acc[r][o] = 0.f;
    for (int c0 = 0; c0 < A.cin; c0 += CVK) {
      __syncthreads();  // the previous chunk's (or image's) reads
      stage_planes<RG>(A, xs, b, x0, y0, c0, CVK, NT);
      for (int t = tid; t < CVK * 9 * CO; t += NT) {
        const int o = t % CO, tap = (t / CO) % 9, c = c0 + t / (9 * CO);
        ws[t] = c < A.cin ? __ldg(A.w + ((8 - tap) * A.cout + o) * A.cin + c) : 0.f;
      }
      __syncthreads();
      const int kn = min(CVK, A.cin - c0);
#pragma unroll 1
      for (int k = 0; k < kn; ++k) {
        float v[CVR + 2][3];
        const float* xp = xs + k * SM::plane + rg * CVR * CVP + lane;
#pragma unroll
        for (int r = 0; r < CVR + 2; ++r)
#pragma unroll
          for (int q = 0; q < 3; ++q) v[r][q] = xp[r * CVP + q];
        const float* wp = ws + k * 9 * CO + cg * COT;
#pragma unroll
        for (int tap = 0; tap < 9; ++tap) {
          float u[CVR];
#pragma unroll
          for (int r = 0; r < CVR; ++r) u[r] = v[r + tap / 3][tap % 3];
          conv_fma<COT>(acc, u, wp + tap * CO);
        }
      }
    }
    conv_store<COT>(A, acc, b, x0 + lane, y0 + rg * CVR, cg * COT);
  }
}

// ---------------------------------------------------------------------------
// BF16 tensor-core forward convolution (mma.sync m16n8k16, FP32 accumulate)
// Block: 8 warps, tile of TR = 8 rows x TC = 32 columns of output pixels; warp
// w owns row w as two M tiles of 16 pixels; N = output channels in tiles of
// 8; K = 9 taps x input channels in steps of 16. The input tile with a
// one-pixel halo and all nine taps of transposed weights are staged once in
// shared memory as BF16, every pixel's (and output channel's) K vector padded
// by 8 elements so that the fragment loads of a warp hit distinct banks.
// ---------------------------------------------------------------------------
constexpr int TR = 8, TC = 32, TCT = 256;

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

template <int CIP, int COP>
struct TcSmem {
  static constexpr int KS = CIP + 8;                     // padded K stride (elements)
  static constexpr int XS = (TR + 2) * (TC + 2) * KS;    // input tile
  static constexpr int WS = 9 * COP * KS;                // weights [tap][co][ci]
  static constexpr size_t bytes = (size_t)(XS + WS) * sizeof(__nv_bfloat16);
};

// CIP: input channels padded to a multiple of 16; COP: output channels padded to a multiple of 8
template <int CIP, int COP>
__global__ void __launch_bounds__(TCT) k_conv_fwd_tc(In2 in, const __nv_bfloat16* __restrict__ wbf /*[9][cin][cout]*/,
                                                     const float* __restrict__ bias, float* __restrict__ out, int cout,
                                                     int n, int h, int wd, int relu) {
  using SM = TcSmem<CIP, COP>;
  constexpr int KS = SM::KS;
  extern __shared__ __align__(16) __nv_bfloat16 tc_smem[];
  __nv_bfloat16* xs = tc_smem;
  __nv_bfloat16* wt = tc_smem + SM::XS;
  const int cin = in.c0 + in.c1;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int x0 = blockIdx.x * TC, y0 = blockIdx.y * TR, b = blockIdx.z;
  // input tile with halo, four channels per item (zero outside the image and
  // in the channel padding)
  constexpr int G4 = CIP / 4;
  for (int t = tid; t < (TR + 2) * (TC + 2) * G4; t += TCT) {
    const int g4 = t % G4, px = t / G4;
    const int ty = px / (TC + 2), tx = px - ty * (TC + 2);
    const int yy = y0 + ty - 1, xx = x0 + tx - 1;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (yy >= 0 && yy < h && xx >= 0 && xx < wd && 4 * g4 < cin) v = in_val4(in, b, yy, xx, h, wd, 4 * g4, cin);
    __nv_bfloat16* d = xs + px * KS + 4 * g4;
    d[0] = __float2bfloat16(v.x);
    d[1] = __float2bfloat16(v.y);
    d[2] = __float2bfloat16(v.z);
    d[3] = __float2bfloat16(v.w);
  }
  // all nine taps of the weights, transposed to [tap][co][ci] (zero padded)
  for (int t = tid; t < 9 * COP * CIP; t += TCT) {
    const int co = t % COP, ci = (t / COP) % CIP, tap = t / (COP * CIP);
    wt[(tap * COP + co) * KS + ci] =
        (ci < cin && co < cout) ? wbf[((long long)tap * cin + ci) * cout + co] : __float2bfloat16(0.f);
  }
  __syncthreads();
  const int g = lane >> 2, tq = lane & 3;
  constexpr int NT = COP / 8;
  float acc[2][NT][4];
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[mt][nt][q] = 0.f;
  const int row = warp;  // output row within the tile
#pragma unroll 1
  for (int tap = 0; tap < 9; ++tap) {
    const int ky = tap / 3, kx = tap - 3 * ky;
    const __nv_bfloat16* wtap = wt + tap * COP * KS;
#pragma unroll
    for (int k0 = 0; k0 < CIP; k0 += 16) {
      uint32_t bb[NT][2];
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        // B[k][n] = w[tap][k0 + k][nt*8 + n], staged as wt[tap][nt*8 + n][k0 + k]
        const __nv_bfloat16* bcol = wtap + (nt * 8 + g) * KS + k0;
        bb[nt][0] = *reinterpret_cast<const uint32_t*>(bcol + 2 * tq);
        bb[nt][1] = *reinterpret_cast<const uint32_t*>(bcol + 2 * tq + 8);
      }
#pragma unroll
      for (int mt = 0; mt < 2; ++mt) {
        // A[m][k] = xs[row + ky][mt*16 + m + kx][k0 + k]
        const __nv_bfloat16* arow0 = xs + ((row + ky) * (TC + 2) + (mt * 16 + g + kx)) * KS + k0;
        const __nv_bfloat16* arow1 = arow0 + 8 * KS;
        uint32_t a[4];
        a[0] = *reinterpret_cast<const uint32_t*>(arow0 + 2 * tq);
        a[1] = *reinterpret_cast<const uint32_t*>(arow1 + 2 * tq);
        a[2] = *reinterpret_cast<const uint32_t*>(arow0 + 2 * tq + 8);
        a[3] = *reinterpret_cast<const uint32_t*>(arow1 + 2 * tq + 8);
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) mma_bf16(acc[mt][nt], a, bb[nt]);
      }
    }
  }
  // D[m][n]: rows g and g + 8, columns 2 tq and 2 tq + 1 of each n tile
  const int yy = y0 + row;
  if (yy >= h) return;
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int xx = x0 + mt * 16 + g + 8 * half;
      if (xx >= wd) continue;
      float* op = out + (((long long)b * h + yy) * wd + xx) * cout;
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int co = nt * 8 + 2 * tq + e;
          if (co < cout) {
            const float v = acc[mt][nt][2 * half + e] + __ldg(bias + co);
            op[co] = relu ? fmaxf(v, 0.f) : v;
          }
        }
    }
}

// ---------------------------------------------------------------------------
// backward
// ---------------------------------------------------------------------------

// Weight gradient: rows of partial sums over pixels p of in[p + tap, ci]
// dpre[p, co] (partial) and of dpre (bpart), which k_reduce_wgrad adds up in
// FP64. A contraction over the pixels, bound by the FP32 pipe once a thread
// owns all nine taps of one input channel and COW outputs: along a pixel row
// it keeps the 3 x 3 window of its channel in registers, so a pixel costs
// three new inputs and COW gradients for 9 COW multiply-adds (the window and
// the gradients of a warp are consecutive words or broadcasts). The thread
// groups of a block share its rows of pixels.
//
// An FP32 sum ends after `chain` pixels (wgrad_shape); `per_row` of them are
// added up beside the running one (TWO: more than one) and leave as the
// thread's part of a row of partials. A row holds 9 x T x COW values at
// (tap T + thread) COW + output, so that a warp's sums are consecutive there.
// On 8 images of 512^2: 48 -> 16 1.51 ms (19 TFLOP/s; staging the bilinear
// input costs as much as the sums), 16 -> 16 0.50 ms, 64 -> 32 at half
// resolution 0.68 ms; the nine layers with their reductions 4.0 ms, a thread
// per weight on 8-pixel patches took 44 ms.
constexpr int WGC = 32;  // columns of a tile
struct WgradArgs {
  In2 in;
  const float* dpre;
  float* partial;
  double* bpart;
  int cin, co, groups, ty, tiles, per_block, n, h, wd;  // ty: rows of a tile
  int chain, per_row;        // pixels of an FP32 sum, sums added into a row of partials
  int rows;                  // rows of partials of a thread group
  int bgroups;               // rows of bpart of a block
};

template <int COW, int NTM, bool TWO>
__global__ void __launch_bounds__(NTM, 512 / NTM) k_wgrad(const WgradArgs A) {
  extern __shared__ __align__(16) float wg_sm[];
  const int cin = A.cin, co = A.co, T = cin * (co / COW), NT = blockDim.x, tid = threadIdx.x;
  const int xrow = (WGC + 2) * cin;
  float* xs = wg_sm;                                         // [ty + 2][34][cin]
  float* ds = wg_sm + ((A.ty + 2) * xrow + 3) / 4 * 4;        // [ty][32][co]
  const int g = tid / T, r = tid - g * T, ci = r % cin, ob = (r / cin) * COW;
  const bool mine = g < A.groups;
  float acc[9][COW];
#pragma unroll
  for (int q = 0; q < 9; ++q)
#pragma unroll
    for (int o = 0; o < COW; ++o) acc[q][o] = 0.f;
  double bsum = 0.0;  // thread t < co * bgroups: sum of dpre[., t % co]
  const int nw = 9 * cin * co;
  float* const rows = A.partial + ((long long)(blockIdx.x * A.groups + g) * A.rows) * nw + (long long)r * COW;
  int done = 0, sums = 0;  // pixels of the current sum, sums written
  float tot[TWO ? 9 : 1][TWO ? COW : 1];  // the row's sums so far
  if constexpr (TWO) {
#pragma unroll
    for (int q = 0; q < 9; ++q)
#pragma unroll
      for (int o = 0; o < COW; ++o) tot[q][o] = 0.f;
  }
  auto flush = [&]() {
    done = 0;
    ++sums;
    if constexpr (TWO) {
#pragma unroll
      for (int q = 0; q < 9; ++q)
#pragma unroll
        for (int o = 0; o < COW; ++o) {
          acc[q][o] += tot[q][o];
          tot[q][o] = acc[q][o];
        }
    }
    if (!TWO || sums % A.per_row == 0) {
      float* out = rows + (long long)((sums - 1) / A.per_row) * nw;
#pragma unroll
      for (int q = 0; q < 9; ++q) {
        float* d = out + q * T * COW;
        if constexpr (COW % 4 == 0) {
#pragma unroll
          for (int o = 0; o < COW; o += 4)
            *reinterpret_cast<float4*>(d + o) = make_float4(acc[q][o], acc[q][o + 1], acc[q][o + 2], acc[q][o + 3]);
        } else {
#pragma unroll
          for (int o = 0; o < COW; ++o) d[o] = acc[q][o];
        }
        if constexpr (TWO) {
#pragma unroll
          for (int o = 0; o < COW; ++o) tot[q][o] = 0.f;
        }
      }
    }
#pragma unroll
    for (int q = 0; q < 9; ++q)
#pragma unroll
      for (int o = 0; o < COW; ++o) acc[q][o] = 0.f;
  };
  const int tx = (A.wd + WGC - 1) / WGC, tyn = (A.h + A.ty - 1) / A.ty;
  const int t1 = min(A.tiles, (int)(blockIdx.x + 1) * A.per_block);
  for (int tile = blockIdx.x * A.per_block; tile < t1; ++tile) {
    const int bx = tile % tx, q = tile / tx, by = q % tyn, b = q / tyn;
    const int x0 = bx * WGC, y0 = by * A.ty;
    __syncthreads();
    const int g4 = (cin + 3) / 4;
    stage<2>((A.ty + 2) * (WGC + 2) * g4, NT, [&](int t) {
      const int k = t % g4, px = t / g4, rr = px / (WGC + 2), yy = y0 + rr - 1, xx = x0 + px - rr * (WGC + 2) - 1;
      if (yy >= 0 && yy < A.h && xx >= 0 && xx < A.wd) return in_val4(A.in, b, yy, xx, A.h, A.wd, 4 * k, cin);
      return make_float4(0.f, 0.f, 0.f, 0.f);
    }, [&](int t, const float4& v) {
      const int k = t % g4, px = t / g4, rr = px / (WGC + 2);
      float* d = xs + rr * xrow + (px - rr * (WGC + 2)) * cin + 4 * k;
      if ((cin & 3) == 0) {
        *reinterpret_cast<float4*>(d) = v;
      } else {
        d[0] = v.x;
        if (4 * k + 1 < cin) d[1] = v.y;
        if (4 * k + 2 < cin) d[2] = v.z;
        if (4 * k + 3 < cin) d[3] = v.w;
      }
    });
    auto dpx = [&](int px, int& ok) -> long long {  // pixel px of the tile
      const int rr = px / WGC, yy = y0 + rr, xx = x0 + px - rr * WGC;
      ok = yy < A.h && xx < A.wd;
      return ((long long)b * A.h + yy) * A.wd + xx;
    };
    if ((co & 3) == 0) {
      stage<4>(A.ty * WGC * (co / 4), NT, [&](int t) {
        int ok;
        const int c4 = t % (co / 4);
        const long long at = dpx(t / (co / 4), ok);
        return ok ? __ldg(reinterpret_cast<const float4*>(A.dpre + at * co + 4 * c4)) : make_float4(0.f, 0.f, 0.f, 0.f);
      }, [&](int t, const float4& v) { *reinterpret_cast<float4*>(ds + 4 * t) = v; });
    } else {
      for (int t = tid; t < A.ty * WGC * co; t += NT) {
        int ok;
        const long long at = dpx(t / co, ok);
        ds[t] = ok ? __ldg(A.dpre + at * co + t % co) : 0.f;
      }
    }
    __syncthreads();
    if (mine) {
      for (int row = g; row < A.ty; row += A.groups) {
        const float* xp = xs + row * xrow + ci;
        const float* dp = ds + row * WGC * co + ob;
        float w[3][3];
#pragma unroll
        for (int ky = 0; ky < 3; ++ky) {
          w[ky][0] = xp[ky * xrow];
          w[ky][1] = xp[ky * xrow + cin];
        }
        const int seg = min(A.chain, WGC);
        for (int xs0 = 0; xs0 < WGC; xs0 += seg) {
#pragma unroll 4
          for (int x = xs0; x < xs0 + seg; ++x) {
#pragma unroll
            for (int ky = 0; ky < 3; ++ky) w[ky][2] = xp[ky * xrow + (x + 2) * cin];
            float d[COW];
            if constexpr (COW % 4 == 0) {
#pragma unroll
              for (int o = 0; o < COW; o += 4) {
                const float4 v = *reinterpret_cast<const float4*>(dp + x * co + o);
                d[o] = v.x;
                d[o + 1] = v.y;
                d[o + 2] = v.z;
                d[o + 3] = v.w;
              }
            } else {
#pragma unroll
              for (int o = 0; o < COW; ++o) d[o] = dp[x * co + o];
            }
#pragma unroll
            for (int q9 = 0; q9 < 9; ++q9)
#pragma unroll
              for (int o = 0; o < COW; ++o) acc[q9][o] = fmaf(w[q9 / 3][q9 % 3], d[o], acc[q9][o]);
#pragma unroll
            for (int ky = 0; ky < 3; ++ky) {
              w[ky][0] = w[ky][1];
              w[ky][1] = w[ky][2];
            }
          }
          done += seg;
          if (done == A.chain) flush();
        }
      }
    }
    // dpre alone: runs of at most `chain` pixels
    if (tid < co * A.bgroups) {
      const int tile_px = A.ty * WGC, run = min(A.chain, tile_px);
      for (int p0 = tid / co * run; p0 < tile_px; p0 += A.bgroups * run) {
        float b = 0.f;
#pragma unroll 8
        for (int px = p0; px < min(p0 + run, tile_px); ++px) b += ds[px * co + tid % co];
        bsum += b;
      }
    }
  }
  if (mine) {
    if (done) flush();
    while (sums < A.rows * A.per_row) flush();  // zeros where the last block has fewer tiles
  }
  if (tid < co * A.bgroups) A.bpart[(long long)blockIdx.x * co * A.bgroups + tid] = bsum;
}

// The rows of partials added in a fixed order: RG row groups of a block (rows k,
// k + RG, ...), then the groups in FP64. Blocks [0, wblocks): the
// weights' sums, from the order of a row (T threads of cow outputs) to
// [tap][ci][co]; the others: the biases'.
//
// Within a group a sum is a pair of floats: Knuth's two-sum gives a value and
// the exact error of every addition, the errors are added up beside it. That
// keeps 2^-47 of the largest partial sum and runs on the FP32 pipe; in FP64
// a thousand rows held that unit for 40 to 100 us a layer (1 x 512^2: 1.12 ms
// for the nine layers' weight gradients, now 0.81). Sums that leave FP32's
// range are formed in FP64.
// A block of NT threads takes RC columns: 8 in 32 row groups; 32 in 8, which
// leaves a quarter of the FP64 additions, where there are at most 256 rows (128
// rows of 9216 sums: 9.1 -> 5.6 us); or 8 in 128, a quarter of the loads one
// after another, where the columns give few blocks (4096 rows of 432 sums:
// 21 -> 14 us).
struct ReduceArgs {
  const float* partial;
  const double* bpart;
  float* out;
  int nrows, brows, cin, co, cow, wblocks;
};
template <int RC, int NT>
__global__ void __launch_bounds__(NT) k_reduce_wgrad(const ReduceArgs A) {
  constexpr int RG = NT / RC;
  __shared__ double sh[NT / 32][RC];
  const int c = threadIdx.x % RC, k = threadIdx.x / RC;
  const bool bias = (int)blockIdx.x >= A.wblocks;
  const int t = ((int)blockIdx.x - (bias ? A.wblocks : 0)) * RC + c;
  const int nw = 9 * A.cin * A.co, nt = bias ? A.co : nw;
  double s = 0.0;
  if (t < nt) {
    if (bias) {
#pragma unroll 8
      for (int b = k; b < A.brows; b += RG) s += A.bpart[(long long)b * A.co + t];
    } else {
      float hi = 0.f, lo = 0.f;
#pragma unroll 16
      for (int b = k; b < A.nrows; b += RG) {
        const float v = A.partial[(long long)b * nw + t];
        const float z = hi + v, w = z - hi;
        lo += (hi - (z - w)) + (v - w);
        hi = z;
      }
      s = (double)hi + (double)lo;
      if (!isfinite(s)) {
        s = 0.0;
        for (int b = k; b < A.nrows; b += RG) s += A.partial[(long long)b * nw + t];
      }
    }
  }
#pragma unroll
  for (int o = 16; o >= RC; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) < RC) sh[threadIdx.x >> 5][c] = s;
  __syncthreads();
  if (k == 0 && t < nt) {
    for (int q = 1; q < NT / 32; ++q) s += sh[q][c];
    int at = nw + t;
    if (!bias) {
      const int T = A.cin * (A.co / A.cow), o = t % A.cow, r = t / A.cow % T, tap = t / (A.cow * T);
      at = (tap * A.cin + r % A.cin) * A.co + r / A.cin * A.cow + o;
    }
    A.out[at] = (float)s;
  }
}

// ---- elementwise passes, four channels per thread (c is a multiple of 4) ----

__device__ __forceinline__ float4 relu_mask4(float4 d, float4 y) {
  return make_float4(y.x > 0.f ? d.x : 0.f, y.y > 0.f ? d.y : 0.f, y.z > 0.f ? d.z : 0.f, y.w > 0.f ? d.w : 0.f);
}

// 2x2 mean pooling (NHWC), h and w of the input
__global__ void __launch_bounds__(UT) k_pool(const float* __restrict__ x, float* __restrict__ y, int n, int h, int w, int c) {
  const int c4 = c / 4, h2 = h / 2, w2 = w / 2;
  for (int q = blockIdx.y; q < n * h2; q += gridDim.y) {
    const int row = q % h2, b = q / h2;
    for (int t = blockIdx.x * UT + threadIdx.x; t < w2 * c4; t += gridDim.x * UT) {
      const int g = t % c4, col = t / c4;
      const float* s = x + (((long long)b * h + 2 * row) * w + 2 * col) * c + 4 * g;
      const float4 p = __ldg((const float4*)s), q = __ldg((const float4*)(s + c));
      const float4 r = __ldg((const float4*)(s + (long long)w * c)), u = __ldg((const float4*)(s + (long long)w * c + c));
      *(float4*)(y + (((long long)b * h2 + row) * w2 + col) * c + 4 * g) =
          make_float4(0.25f * (p.x + q.x + r.x + u.x), 0.25f * (p.y + q.y + r.y + u.y), 0.25f * (p.z + q.z + r.z + u.z),
                      0.25f * (p.w + q.w + r.w + u.w));
    }
  }
}

// dx (h, w) = relu mask of y (dx + pool adjoint of dy (h/2, w/2))
__global__ void __launch_bounds__(UT) k_pool_bwd_add(const float* __restrict__ dy, float* __restrict__ dx,
                                                     const float* __restrict__ y, int n, int h, int w, int c) {
  const int c4 = c / 4;
  for (int q = blockIdx.y; q < n * h; q += gridDim.y) {
    const int row = q % h, b = q / h;
    for (int t = blockIdx.x * UT + threadIdx.x; t < w * c4; t += gridDim.x * UT) {
      const int g = t % c4, col = t / c4;
      const long long at = (((long long)b * h + row) * w + col) * c + 4 * g;
      const float4 e = __ldg((const float4*)(dy + (((long long)b * (h / 2) + row / 2) * (w / 2) + col / 2) * c + 4 * g));
      float4 v = *(const float4*)(dx + at);
      v.x += 0.25f * e.x;
      v.y += 0.25f * e.y;
      v.z += 0.25f * e.z;
      v.w += 0.25f * e.w;
      *(float4*)(dx + at) = relu_mask4(v, __ldg((const float4*)(y + at)));
    }
  }
}

// weights with which coarse index k (of m) feeds fine indices 2k-1 .. 2k+2
// under bilinear doubling (the clamped edge adds the outer quarter back)
__device__ __forceinline__ void up_adj_weights(int k, int m, float (&wgt)[4]) {
  wgt[0] = k >= 1 ? 0.25f : 0.f;
  wgt[1] = k == 0 ? 1.f : 0.75f;
  wgt[2] = k == m - 1 ? 1.f : 0.75f;
  wgt[3] = k + 1 <= m - 1 ? 0.25f : 0.f;
}

// d (h/2, w/2) = relu mask of y (adjoint of bilinear doubling of dfull (h, w))
__global__ void __launch_bounds__(UT) k_up_bwd(const float* __restrict__ dfull, float* __restrict__ d,
                                               const float* __restrict__ y, int n, int h, int w, int c) {
  const int h0 = h / 2, w0 = w / 2, c4 = c / 4;
  for (int q = blockIdx.y; q < n * h0; q += gridDim.y) {
    const int k = q % h0, b = q / h0;
    float wy[4];
    up_adj_weights(k, h0, wy);
    for (int t = blockIdx.x * UT + threadIdx.x; t < w0 * c4; t += gridDim.x * UT) {
      const int g = t % c4, l = t / c4;
      float wx[4];
      up_adj_weights(l, w0, wx);
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        if (wy[a] == 0.f) continue;
        const float* row = dfull + (((long long)b * h + 2 * k - 1 + a) * w) * c + 4 * g;
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (wx[e] != 0.f) {
            const float4 v = __ldg((const float4*)(row + (long long)(2 * l - 1 + e) * c));
            s.x = fmaf(wx[e], v.x, s.x);
            s.y = fmaf(wx[e], v.y, s.y);
            s.z = fmaf(wx[e], v.z, s.z);
            s.w = fmaf(wx[e], v.w, s.w);
          }
        acc.x = fmaf(wy[a], s.x, acc.x);
        acc.y = fmaf(wy[a], s.y, acc.y);
        acc.z = fmaf(wy[a], s.z, acc.z);
        acc.w = fmaf(wy[a], s.w, acc.w);
      }
      const long long at = (((long long)b * h0 + k) * w0 + l) * c + 4 * g;
      *(float4*)(d + at) = relu_mask4(acc, __ldg((const float4*)(y + at)));
    }
  }
}

// dy = scale (y - tscale t) (scale = 2 / batch), and the sum of (y - tscale t)^2
__global__ void __launch_bounds__(256) k_mse(const float* __restrict__ y, const float* __restrict__ t, float* __restrict__ dy,
                                             long long n, float scale, float tscale, RedBuf red, double* out) {
  double acc = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float d = y[i] - tscale * t[i];
    dy[i] = scale * d;
    acc += (double)d * (double)d;
  }
  double v[1] = {acc};
  grid_reduce<1>(v, red, FIN_STORE, out);
}

__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                       long long n, float lr, float b1, float b2, float eps, float c1, float c2) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi * c1) / (sqrtf(vi * c2) + eps);
  }
}

__global__ void k_to_bf16(const float* __restrict__ a, __nv_bfloat16* __restrict__ b, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    b[i] = __float2bfloat16(a[i]);
}

// He-normal initial weights (std sqrt(2 / (9 cin))), zero biases, from a
// counter-based hash of (seed, index) and the Box-Muller transform
__global__ void k_init_params(float* p, long long off, long long nw, int cin, int cout, unsigned long long seed) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nw + cout; i += (long long)gridDim.x * blockDim.x) {
    if (i >= nw) { p[off + i] = 0.f; continue; }
    unsigned long long z = (seed + (unsigned long long)(off + i)) * 0x9E3779B97F4A7C15ull;
    z ^= z >> 30; z *= 0xBF58476D1CE4E5B9ull; z ^= z >> 27; z *= 0x94D049BB133111EBull; z ^= z >> 31;
    const double u1 = ((z >> 11) + 1.0) * (1.0 / 9007199254740993.0);
    unsigned long long z2 = z * 0x9E3779B97F4A7C15ull + 1442695040888963407ull;
    z2 ^= z2 >> 31;
    const double u2 = (z2 >> 11) * (1.0 / 9007199254740992.0);
    const double nrm = sqrt(-2.0 * log(u1)) * cos(6.283185307179586 * u2);
    p[off + i] = (float)(nrm * sqrt(2.0 / (9.0 * cin)));
  }
}

static unsigned grid_for(long long n, int per = UT) {
  long long b = (n + per - 1) / per;
  if (b > 4096) b = 4096;
  return (unsigned)(b < 1 ? 1 : b);
}

// grid of the elementwise passes: one row of an image per y
static dim3 row_grid(int items, int rows) { return dim3((items + UT - 1) / UT, std::min(rows, 65535)); }

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

// shared memory of an FP32 forward convolution of cin channels
template <int COT, int CG, int RG>
static size_t fwd_smem(int cin) {
  return ((size_t)(cin + 3) / 4 * 4 * ConvSmem<RG>::plane + 9ull * cin * COT * CG) * sizeof(float);
}
// The limit belongs to the kernel, not to a launch: it is set once, for the
// widest layer that takes the instance. Set per launch, another thread's
// narrower layer could lower it between this thread's call and its launch.
template <int COT, int CG, int RG>
static void allow_fwd(int cin) {
  GKB_CUDA(cudaFuncSetAttribute(k_conv_fwd<COT, CG, RG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)fwd_smem<COT, CG, RG>(cin)));
}

void Unet::init(int cin, int k1, int k2, int cout, unsigned long long seed, cudaStream_t s) {
  c_in = cin; c1 = k1; c2 = k2; c_out = cout; stream = s;
  if (!(cin >= 1 && cin <= 16 && k1 == 16 && k2 == 32 && cout >= 1 && cout <= 3))
    throw Error{GKB_ERR_INVALID_ARG, "supported U-Net: 1..16 inputs, 16/32 channels, 1..3 outputs"};
  const int shapes[9][2] = {{cin, k1}, {k1, k1}, {k1, k2}, {k2, k2}, {k2, k2}, {k2, k2}, {2 * k2, k2}, {k2 + k1, k1}, {k1, cout}};
  layers.clear();
  long long off = 0;
  for (auto& sh : shapes) {
    layers.push_back(ConvLayer{sh[0], sh[1], off});
    off += 9LL * sh[0] * sh[1] + sh[1];
  }
  nparams = off;
  params.alloc(nparams);
  grads.alloc(nparams);
  adam_m.alloc(nparams);
  adam_v.alloc(nparams);
  params_bf16.alloc(nparams);
  for (const ConvLayer& L : layers) {
    k_init_params<<<grid_for(L.nw() + L.cout), UT, 0, s>>>(params.p, L.off, L.nw(), L.cin, L.cout, seed);
    GKB_CUDA(cudaGetLastError());
  }
  red_partial.alloc(4096 * 4 + 64);
  red_ticket.alloc(1);
  loss_dev.alloc(4);
  // the tensor-core convolutions stage all nine weight taps (up to 80 KB)
  GKB_CUDA(cudaFuncSetAttribute(k_conv_fwd_tc<16, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcSmem<16, 8>::bytes));
  GKB_CUDA(cudaFuncSetAttribute(k_conv_fwd_tc<16, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcSmem<16, 16>::bytes));
  GKB_CUDA(cudaFuncSetAttribute(k_conv_fwd_tc<16, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcSmem<16, 32>::bytes));
  GKB_CUDA(cudaFuncSetAttribute(k_conv_fwd_tc<32, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcSmem<32, 32>::bytes));
  GKB_CUDA(cudaFuncSetAttribute(k_conv_fwd_tc<48, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcSmem<48, 16>::bytes));
  GKB_CUDA(cudaFuncSetAttribute(k_conv_fwd_tc<64, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcSmem<64, 32>::bytes));
  allow_fwd<16, 1, 4>(16);
  allow_fwd<16, 2, 4>(16);
  allow_fwd<8, 2, 4>(48);
  allow_fwd<8, 2, 1>(48);
  allow_fwd<8, 4, 2>(64);
  allow_fwd<8, 4, 1>(64);
  for (auto f : {k_wgrad<4, 256, false>, k_wgrad<4, 256, true>, k_wgrad<4, 512, false>, k_wgrad<4, 512, true>})
    GKB_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024));
  bf16_stale = true;
  adam_t = 0;
}

void Unet::ensure(UnetAct& A, int n, int h, int w) const {
  if (h % 4 || w % 4 || n < 1 || h < 4 || w < 4) throw Error{GKB_ERR_INVALID_ARG, "U-Net images need sides divisible by 4"};
  if (n == A.n && h == A.h && w == A.w) return;
  const long long P = (long long)n * h * w, P2 = P / 4, P4 = P / 16;
  A.a1.alloc(P * c1); A.s1.alloc(P * c1); A.e1.alloc(P * c1); A.y.alloc(P * c_out);
  A.p1.alloc(P2 * c1); A.b1.alloc(P2 * c2); A.s2.alloc(P2 * c2); A.d1.alloc(P2 * c2);
  A.p2.alloc(P4 * c2); A.c1a.alloc(P4 * c2); A.c2a.alloc(P4 * c2);
  A.n = n; A.h = h; A.w = w;
}

void Unet::refresh_bf16(cudaStream_t s) {
  ProfScope ps_(GKB_KC_UNET, s, nparams);
  k_to_bf16<<<grid_for(nparams), UT, 0, s>>>(params.p, params_bf16.p, nparams);
  GKB_CUDA(cudaGetLastError());
  bf16_stale = false;
}

// an FP32 convolution's grid; tall tiles (RG row groups) where they give every
// SM a block, else one-warp-high ones (a 128^2 image has 32 tall tiles)
static dim3 conv_grid(const ConvArgs& A, int rg) {
  return dim3((A.wd + 31) / 32, (A.h + CVR * rg - 1) / (CVR * rg), std::min(A.n, 65535));
}
static bool fills(dim3 g) { return (long long)g.x * g.y * g.z >= 152; }

template <int COT, int CG, int RG>
static void launch_fwd(const ConvArgs& A, cudaStream_t s) {
  k_conv_fwd<COT, CG, RG><<<conv_grid(A, RG), 32 * CG * RG, fwd_smem<COT, CG, RG>(A.cin), s>>>(A);
}
template <int COT, int CG, int RG>
static void conv_fwd32(const ConvArgs& A, cudaStream_t s) {
  if (RG == 1 || fills(conv_grid(A, RG))) launch_fwd<COT, CG, RG>(A, s);
  else launch_fwd<COT, CG, 1>(A, s);
  GKB_CUDA(cudaGetLastError());
}
template <int COT, int CG, int RG>
static void conv_bwd32(const ConvArgs& A, cudaStream_t s) {
  const dim3 g = conv_grid(A, RG);
  if (fills(g)) k_conv_bwd<COT, CG, RG><<<g, 32 * CG * RG, 0, s>>>(A);
  else k_conv_bwd<COT, CG, 1><<<conv_grid(A, 1), 32 * CG, 0, s>>>(A);
  GKB_CUDA(cudaGetLastError());
}

static void conv_fwd(const Unet& U, int li, In2 in, float* out, int n, int h, int w, int relu, bool tc,
                     cudaStream_t s) {
  const ConvLayer& L = U.layers[li];
  const float* wp = U.params.p + L.off;
  const float* bp = wp + L.nw();
  const long long P = (long long)n * h * w;
  ProfScope ps_(GKB_KC_UNET, s, P);
  if (tc) {
    const __nv_bfloat16* wb = U.params_bf16.p + L.off;
    dim3 grid((w + TC - 1) / TC, (h + TR - 1) / TR, n);
    const int cin = L.cin;
#define GKB_TC(CI, CO) \
  k_conv_fwd_tc<CI, CO><<<grid, TCT, TcSmem<CI, CO>::bytes, s>>>(in, wb, bp, out, L.cout, n, h, w, relu)
    if (cin <= 16 && L.cout <= 8) GKB_TC(16, 8);
    else if (cin <= 16 && L.cout <= 16) GKB_TC(16, 16);
    else if (cin <= 16) GKB_TC(16, 32);
    else if (cin <= 32) GKB_TC(32, 32);
    else if (cin <= 48) GKB_TC(48, 16);
    else GKB_TC(64, 32);
#undef GKB_TC
  } else {
    // outputs per thread and groups by layer: as many blocks per SM as the
    // staged channels leave room for
    const ConvArgs A{in, wp, bp, out, nullptr, nullptr, L.cout, L.cin, L.cout, relu, n, h, w};
    if (L.cout <= 4) conv_fwd32<4, 1, 4>(A, s);
    else if (L.cout == 16 && L.cin <= 16) conv_fwd32<16, 1, 4>(A, s);
    else if (L.cout == 16) conv_fwd32<8, 2, 4>(A, s);
    else if (L.cin <= 16) conv_fwd32<16, 2, 4>(A, s);
    else conv_fwd32<8, 4, 2>(A, s);
  }
  GKB_CUDA(cudaGetLastError());
}

const float* Unet::forward(UnetAct& A, const float* x, int n, int h, int w, bool tc, cudaStream_t s) {
  ensure(A, n, h, w);
  if (tc && bf16_stale) refresh_bf16(s);
  const int h2 = h / 2, w2 = w / 2, h4 = h / 4, w4 = w / 4;
  conv_fwd(*this, 0, make_in(x, c_in), A.a1.p, n, h, w, 1, tc, s);
  conv_fwd(*this, 1, make_in(A.a1.p, c1), A.s1.p, n, h, w, 1, tc, s);
  { ProfScope ps_(GKB_KC_UNET, s); k_pool<<<row_grid(w2 * c1 / 4, n * h2), UT, 0, s>>>(A.s1.p, A.p1.p, n, h, w, c1); }
  conv_fwd(*this, 2, make_in(A.p1.p, c1), A.b1.p, n, h2, w2, 1, tc, s);
  conv_fwd(*this, 3, make_in(A.b1.p, c2), A.s2.p, n, h2, w2, 1, tc, s);
  { ProfScope ps_(GKB_KC_UNET, s); k_pool<<<row_grid(w4 * c2 / 4, n * h4), UT, 0, s>>>(A.s2.p, A.p2.p, n, h2, w2, c2); }
  conv_fwd(*this, 4, make_in(A.p2.p, c2), A.c1a.p, n, h4, w4, 1, tc, s);
  conv_fwd(*this, 5, make_in(A.c1a.p, c2), A.c2a.p, n, h4, w4, 1, tc, s);
  conv_fwd(*this, 6, make_in(A.c2a.p, c2, 1, A.s2.p, c2), A.d1.p, n, h2, w2, 1, tc, s);
  conv_fwd(*this, 7, make_in(A.d1.p, c2, 1, A.s1.p, c1), A.e1.p, n, h, w, 1, tc, s);
  conv_fwd(*this, 8, make_in(A.e1.p, c1), A.y.p, n, h, w, 0, tc, s);
  return A.y.p;
}

// Launch shape of layer L's weight gradient on n images of h x w, N pixels.
//
// Rounding: an FP32 sum of F terms leaves an error of about sqrt(F / 2) units
// of its last place, and the sums of R / F of them in a row sqrt(R / (2 F)).
// The bound kept is that of sums over 8 pixels added up by 304 blocks,
// 8 + N / 2432 for F: F is the largest power of two below 0.65 of it, which
// leaves room for the additions into a row and for neighbouring terms that are
// not independent, at least 8. A row takes R = N / 1280 pixels of a thread group
// (a power of two, at least F; up to four groups count), so that 640 to 1280
// rows of a group are written and added up.
// One sum per thread over all its pixels (128 to 2048) was up to five times as
// far off. Training steps against it: 1 x 64^2 0.74 -> 0.70 ms, 1 x 128^2 0.77
// -> 0.75, 1 x 256^2 0.94 -> 0.99, 8 x 96^2 1.07 -> 1.14, 1 x 512^2 1.89 -> 1.79,
// 8 x 512^2 9.97 -> 9.72.
constexpr int WG_ROWS = 1280;
// Outputs per thread: 4 (two sums of each: 16 warps of 128 registers per SM; 64
// -> 32 takes blocks of 512 threads), 2 where so few channels leave threads idle.
static int wgrad_cow(const ConvLayer& L) {
  if (L.cout % 8) return L.cout;
  return L.cin * L.cout / 4 < 32 ? 2 : 4;
}
static WgradArgs wgrad_shape(const ConvLayer& L, int n, int h, int w) {
  WgradArgs A{};
  A.cin = L.cin;
  A.co = L.cout;
  A.n = n;
  A.h = h;
  A.wd = w;
  const int T = L.cin * (L.cout / wgrad_cow(L));
  A.groups = std::max(1, std::min(8, 256 / T));
  // rows of a tile: four (a halo of two more), or one of each group where that
  // leaves SMs without a block
  A.ty = std::max(4, A.groups);
  auto tiles = [&] { return n * ((w + WGC - 1) / WGC) * ((h + A.ty - 1) / A.ty); };
  if (tiles() < 152) A.ty = A.groups;
  A.tiles = tiles();
  const long long N = (long long)n * h * w;
  A.chain = 8;
  while (2 * A.chain <= 0.65 * (8 + N / 2432.0)) A.chain *= 2;
  const int px = WGC * A.ty / A.groups;  // pixels of a tile per thread
  long long row = A.chain;  // pixels of a row of partials
  while (row * WG_ROWS * std::min(A.groups, 4) < N) row *= 2;
  A.per_row = (int)(row / A.chain);
  A.per_block = (int)std::max(1LL, row / px);
  A.rows = (int)std::max(1LL, px / row);
  const int runs = (WGC * A.ty + A.chain - 1) / A.chain;  // runs of dpre sums in a tile
  A.bgroups = std::min(runs, std::max(1, T * A.groups / L.cout));
  return A;
}

// weight gradient of layer li into grads (two deterministic passes)
static void conv_bwd_w(Unet& U, int li, In2 in, const float* dpre, int n, int h, int w) {
  const ConvLayer& L = U.layers[li];
  WgradArgs A = wgrad_shape(L, n, h, w);
  A.in = in;
  A.dpre = dpre;
  const int nblk = (A.tiles + A.per_block - 1) / A.per_block;
  const size_t np = (size_t)nblk * A.groups * A.rows * L.nw(), nb = (size_t)nblk * A.bgroups * L.cout;
  if (U.wpart.n < np) U.wpart.alloc(np);
  if (U.bpart.n < nb) U.bpart.alloc(nb);
  A.partial = U.wpart.p;
  A.bpart = U.bpart.p;
  const int cow = wgrad_cow(L), T = L.cin * (L.cout / cow);
  const int nt = (std::max(T * A.groups, L.cout) + 31) / 32 * 32;
  const size_t tile = ((size_t)(A.ty + 2) * (WGC + 2) * L.cin + 3) / 4 * 4 + (size_t)A.ty * WGC * L.cout;
  const size_t sm = tile * sizeof(float);
  cudaStream_t s = U.stream;
  ProfScope ps_(GKB_KC_UNET, s, (long long)n * h * w);
  const bool two = A.per_row > 1;
#define GKB_WG(COW, NTM)                                  \
  if (two) k_wgrad<COW, NTM, true><<<nblk, nt, sm, s>>>(A); \
  else k_wgrad<COW, NTM, false><<<nblk, nt, sm, s>>>(A)
  if (cow == 4 && nt > 256) { GKB_WG(4, 512); }
  else if (cow == 4) { GKB_WG(4, 256); }
  else if (cow == 3) { GKB_WG(3, 256); }
  else if (cow == 2) { GKB_WG(2, 256); }
  else { GKB_WG(1, 256); }
#undef GKB_WG
  ReduceArgs R{U.wpart.p, U.bpart.p, U.grads.p + L.off, nblk * A.groups * A.rows, nblk * A.bgroups, L.cin, L.cout, cow, 0};
  const int rc = R.nrows <= 256 ? 32 : 8;
  R.wblocks = (int)((L.nw() + rc - 1) / rc);
  const int blocks = R.wblocks + (L.cout + rc - 1) / rc;
  if (rc == 32) k_reduce_wgrad<32, 256><<<blocks, 256, 0, s>>>(R);
  else if (blocks < 304) k_reduce_wgrad<8, 1024><<<blocks, 1024, 0, s>>>(R);
  else k_reduce_wgrad<8, 256><<<blocks, 256, 0, s>>>(R);
  GKB_CUDA(cudaGetLastError());
}

// d_in of layer li (all input channels), split at c0 into d0 / d1; with mask,
// d0 passes the ReLU that produced it
static void conv_bwd_data(Unet& U, int li, const float* dpre, int c0, float* d0, float* d1, const float* mask, int n,
                          int h, int w) {
  const ConvLayer& L = U.layers[li];
  ProfScope ps_(GKB_KC_UNET, U.stream, (long long)n * h * w);
  const ConvArgs A{make_in(dpre, L.cout), U.params.p + L.off, nullptr, d0, d1, mask, c0, L.cout, L.cin, 0, n, h, w};
  if (L.cin == 16) conv_bwd32<16, 1, 8>(A, U.stream);
  else if (L.cin == 32) conv_bwd32<16, 2, 4>(A, U.stream);
  else if (L.cin == 48) conv_bwd32<16, 3, 4>(A, U.stream);
  else if (L.cin == 64) conv_bwd32<16, 4, 4>(A, U.stream);
  else throw Error{GKB_ERR_INVALID_ARG, "unsupported convolution shape in backward"};
}

double Unet::loss_grad(const float* x, const float* t, int n, int h, int w) {
  cudaStream_t s = stream;
  forward(act, x, n, h, w, false, s);
  if (n != gn || h != gh || w != gw) {
    const long long P = (long long)n * h * w, P2 = P / 4, P4 = P / 16;
    g_full0.alloc(P * c2); g_full1.alloc(P * c2); g_e.alloc(P * c1);
    g_half0.alloc(P2 * c2); g_half1.alloc(P2 * c2);
    g_q0.alloc(P4 * c2); g_q1.alloc(P4 * c2);
    gn = n; gh = h; gw = w;
  }
  float *a1 = act.a1.p, *s1 = act.s1.p, *p1 = act.p1.p, *b1 = act.b1.p, *s2 = act.s2.p, *p2 = act.p2.p;
  float *c1a = act.c1a.p, *c2a = act.c2a.p, *d1 = act.d1.p, *e1 = act.e1.p, *y = act.y.p;
  const int h2 = h / 2, w2 = w / 2, h4 = h / 4, w4 = w / 4;
  const long long P = (long long)n * h * w;
  RedBuf red{red_partial.p, red_ticket.p};
  // dy = y - t (into g_e with c_out channels: g_e holds P * c1 >= P * c_out)
  float* dy = g_e.p;
  {
    ProfScope ps_(GKB_KC_UNET, s);
    k_mse<<<grid_for(P * c_out), 256, 0, s>>>(y, t, dy, P * c_out, 2.f / (float)n, target_scale, red, loss_dev.p);
  }
  // out layer (no ReLU): input e1
  conv_bwd_w(*this, 8, make_in(e1, c1), dy, n, h, w);
  float* de1 = g_full1.p;  // P * c1
  conv_bwd_data(*this, 8, dy, c1, de1, nullptr, e1, n, h, w);
  // e1 = relu(conv([up(d1), s1]))
  conv_bwd_w(*this, 7, make_in(d1, c2, 1, s1, c1), de1, n, h, w);
  float* du1 = g_full0.p;     // P * c2 (gradient of up(d1))
  float* ds1 = g_e.p;         // P * c1 (dy no longer needed)
  conv_bwd_data(*this, 7, de1, c2, du1, ds1, nullptr, n, h, w);
  float* dd1 = g_half0.p;     // P2 * c2
  k_up_bwd<<<row_grid(w2 * c2 / 4, n * h2), UT, 0, s>>>(du1, dd1, d1, n, h, w, c2);
  // d1 = relu(conv([up(c2a), s2]))
  conv_bwd_w(*this, 6, make_in(c2a, c2, 1, s2, c2), dd1, n, h2, w2);
  float* du2 = g_full1.p;     // P2 * c2 (reuse)
  float* ds2 = g_half1.p;     // P2 * c2
  conv_bwd_data(*this, 6, dd1, c2, du2, ds2, nullptr, n, h2, w2);
  float* dc2 = g_q0.p;        // P4 * c2
  k_up_bwd<<<row_grid(w4 * c2 / 4, n * h4), UT, 0, s>>>(du2, dc2, c2a, n, h2, w2, c2);
  conv_bwd_w(*this, 5, make_in(c1a, c2), dc2, n, h4, w4);
  float* dc1 = g_q1.p;
  conv_bwd_data(*this, 5, dc2, c2, dc1, nullptr, c1a, n, h4, w4);
  conv_bwd_w(*this, 4, make_in(p2, c2), dc1, n, h4, w4);
  float* dp2 = g_q0.p;
  conv_bwd_data(*this, 4, dc1, c2, dp2, nullptr, nullptr, n, h4, w4);
  k_pool_bwd_add<<<row_grid(w2 * c2 / 4, n * h2), UT, 0, s>>>(dp2, ds2, s2, n, h2, w2, c2);
  conv_bwd_w(*this, 3, make_in(b1, c2), ds2, n, h2, w2);
  float* db1 = g_half0.p;
  conv_bwd_data(*this, 3, ds2, c2, db1, nullptr, b1, n, h2, w2);
  conv_bwd_w(*this, 2, make_in(p1, c1), db1, n, h2, w2);
  float* dp1 = g_half1.p;     // P2 * c1
  conv_bwd_data(*this, 2, db1, c1, dp1, nullptr, nullptr, n, h2, w2);
  k_pool_bwd_add<<<row_grid(w * c1 / 4, n * h), UT, 0, s>>>(dp1, ds1, s1, n, h, w, c1);
  conv_bwd_w(*this, 1, make_in(a1, c1), ds1, n, h, w);
  float* da1 = g_full1.p;
  conv_bwd_data(*this, 1, ds1, c1, da1, nullptr, a1, n, h, w);
  conv_bwd_w(*this, 0, make_in(x, c_in), da1, n, h, w);
  GKB_CUDA(cudaGetLastError());
  double loss = 0.0;
  GKB_CUDA(cudaMemcpyAsync(&loss, loss_dev.p, sizeof(double), cudaMemcpyDeviceToHost, s));
  GKB_CUDA(cudaStreamSynchronize(s));
  return loss / n;
}

void Unet::adam(float lr, float beta1, float beta2, float eps) {
  adam_t += 1;
  const float c1f = (float)(1.0 / (1.0 - pow((double)beta1, (double)adam_t)));
  const float c2f = (float)(1.0 / (1.0 - pow((double)beta2, (double)adam_t)));
  ProfScope ps_(GKB_KC_UNET, stream, nparams);
  k_adam<<<grid_for(nparams), UT, 0, stream>>>(params.p, grads.p, adam_m.p, adam_v.p, nparams, lr, beta1, beta2, eps, c1f, c2f);
  GKB_CUDA(cudaGetLastError());
  bf16_stale = true;
}

void Unet::train(const float* x_img, const float* t_img, long long count, int h, int w, int batch, int steps, float lr,
                 unsigned long long seed, double* losses) {
  if (count < 1 || batch < 1 || batch > count || steps < 0 || !(lr > 0))
    throw Error{GKB_ERR_INVALID_ARG, "training needs 1 <= batch <= count, steps >= 0 and lr > 0"};
  const long long xs = (long long)h * w * c_in, ts = (long long)h * w * c_out;
  if (xb.n != (size_t)(batch * xs)) xb.alloc((size_t)batch * xs);
  if (tb.n != (size_t)(batch * ts)) tb.alloc((size_t)batch * ts);
  std::vector<long long> order(count);
  for (long long i = 0; i < count; ++i) order[i] = i;
  std::mt19937_64 rng(seed);
  long long pos = count;  // forces a shuffle before the first batch
  for (int it = 0; it < steps; ++it) {
    for (int b = 0; b < batch; ++b) {
      if (pos == count) {
        std::shuffle(order.begin(), order.end(), rng);
        pos = 0;
      }
      const long long k = order[pos++];
      GKB_CUDA(cudaMemcpyAsync(xb.p + b * xs, x_img + k * xs, xs * sizeof(float), cudaMemcpyDeviceToDevice, stream));
      GKB_CUDA(cudaMemcpyAsync(tb.p + b * ts, t_img + k * ts, ts * sizeof(float), cudaMemcpyDeviceToDevice, stream));
    }
    const double l = loss_grad(xb.p, tb.p, batch, h, w);
    if (losses) losses[it] = l;
    adam(lr, 0.9f, 0.999f, 1e-8f);
  }
  GKB_CUDA(cudaStreamSynchronize(stream));
}

// ---------------------------------------------------------------------------
// the network as a coarse correction on a 2D MAC level
// ---------------------------------------------------------------------------

// image (ny, nx, 3): west u face and south v face of each cell scaled by
// sqrt(nx ny / ||b||^2), and log viscosity
template <typename T>
__global__ void k_mac_to_img(Lvl L, const T* __restrict__ b, const double* __restrict__ nrm, float* __restrict__ img) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
  if (i >= L.n[0] || j >= L.n[1]) return;
  const double nr2 = nrm[0];
  const double sc = nr2 > 0.0 ? sqrt((double)L.n[0] * L.n[1] / nr2) : 0.0;
  const long long c = cix(L, i, j, 0);
  float* o = img + ((long long)j * L.n[0] + i) * 3;
  o[0] = face_active<0>(L, i, j, 0) ? (float)((double)b[L.off[0] + c] * sc) : 0.f;
  o[1] = face_active<1>(L, i, j, 0) ? (float)((double)b[L.off[1] + c] * sc) : 0.f;
  const T* mu = MuPtr<T>::get(L);
  o[2] = (float)log(mu ? (double)mu[c] : L.mu0);
}

// x on every face of the level: the network output scaled back, zero on the
// faces that are not unknowns and on east / north boundary faces
template <typename T>
__global__ void k_img_to_mac(Lvl L, const float* __restrict__ y, const double* __restrict__ nrm, float inv_tscale,
                             T* __restrict__ x) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
  if (i > L.n[0] || j > L.n[1]) return;
  const double nr2 = nrm[0];
  const double sc = nr2 > 0.0 ? sqrt(nr2 / ((double)L.n[0] * L.n[1])) * inv_tscale : 0.0;
  const long long c = cix(L, i, j, 0);
  const bool in = i < L.n[0] && j < L.n[1];
  if (j < L.n[1]) {  // u face (i, j), i <= nx
    const bool a = in && face_active<0>(L, i, j, 0);
    x[L.off[0] + c] = a ? (T)((double)y[((long long)j * L.n[0] + i) * 2 + 0] * sc) : (T)0;
  }
  if (i < L.n[0]) {  // v face (i, j), j <= ny
    const bool a = in && face_active<1>(L, i, j, 0);
    x[L.off[1] + c] = a ? (T)((double)y[((long long)j * L.n[0] + i) * 2 + 1] * sc) : (T)0;
  }
}

// (xs - xk) on the west u / south v face of every cell, scaled like k_mac_to_img
__global__ void k_err_to_img(Lvl L, const double* __restrict__ xs, const double* __restrict__ xk,
                             const double* __restrict__ nrm, float* __restrict__ img) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
  if (i >= L.n[0] || j >= L.n[1]) return;
  const double nr2 = nrm[0];
  const double sc = nr2 > 0.0 ? sqrt((double)L.n[0] * L.n[1] / nr2) : 0.0;
  const long long c = cix(L, i, j, 0);
  float* o = img + ((long long)j * L.n[0] + i) * 2;
  const long long cu = L.off[0] + c, cv = L.off[1] + c;
  o[0] = face_active<0>(L, i, j, 0) ? (float)((xs[cu] - xk[cu]) * sc) : 0.f;
  o[1] = face_active<1>(L, i, j, 0) ? (float)((xs[cv] - xk[cv]) * sc) : 0.f;
}

template <typename T>
void mac_to_img(const Lvl& L, const T* b, const double* nrm, float* img, cudaStream_t s) {
  ProfScope ps_(GKB_KC_UNET, s, (long long)L.n[0] * L.n[1]);
  k_mac_to_img<T><<<dim3((L.n[0] + 31) / 32, (L.n[1] + 7) / 8), dim3(32, 8), 0, s>>>(L, b, nrm, img);
  GKB_CUDA(cudaGetLastError());
}
template void mac_to_img<double>(const Lvl&, const double*, const double*, float*, cudaStream_t);
template void mac_to_img<float>(const Lvl&, const float*, const double*, float*, cudaStream_t);

void err_to_img(const Lvl& L, const double* xs, const double* xk, const double* nrm, float* img, cudaStream_t s) {
  ProfScope ps_(GKB_KC_UNET, s, (long long)L.n[0] * L.n[1]);
  k_err_to_img<<<dim3((L.n[0] + 31) / 32, (L.n[1] + 7) / 8), dim3(32, 8), 0, s>>>(L, xs, xk, nrm, img);
  GKB_CUDA(cudaGetLastError());
}

// x *= omega, omega = d[0] / d[1] when d[1] > 0, else 0
template <typename T>
__global__ void k_scale_step(T* __restrict__ x, long long n, const double* __restrict__ d) {
  const double den = d[1];
  const T w = (T)(den > 0.0 && isfinite(den) && isfinite(d[0]) ? d[0] / den : 0.0);
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
    x[t] *= w;
}

template <typename T>
void unet_correct(Unet& U, UnetAct& A, const Lvl& L, const T* b, T* x, T* q, float* img_in, double* nrm,
                  const RedBuf& red, cudaStream_t s) {
  if (L.dim != 2) throw Error{GKB_ERR_INVALID_ARG, "the learned correction is 2D only"};
  Ops<T>::dot(L.nvel, b, b, red, FIN_STORE, nrm, s);
  const dim3 blk(32, 8);
  mac_to_img<T>(L, b, nrm, img_in, s);
  const float* y = U.forward(A, img_in, 1, L.n[1], L.n[0], true, s);
  {
    ProfScope ps_(GKB_KC_UNET, s, (long long)L.n[0] * L.n[1]);
    k_img_to_mac<T><<<dim3((L.n[0] + 32) / 32, (L.n[1] + 8) / 8), blk, 0, s>>>(L, y, nrm, 1.f / U.target_scale, x);
  }
  // energy-optimal step along the network's direction
  Ops<T>::apply(L, 1, x, q, s);
  Ops<T>::dot2(L.nvel, b, x, q, red, FIN_STORE, nrm + 4, s);
  {
    ProfScope ps_(GKB_KC_UNET, s, L.nvel);
    k_scale_step<T><<<grid_for(L.nvel), UT, 0, s>>>(x, L.nvel, nrm + 4);
  }
  GKB_CUDA(cudaGetLastError());
}

template void unet_correct<double>(Unet&, UnetAct&, const Lvl&, const double*, double*, double*, float*, double*,
                                   const RedBuf&, cudaStream_t);
template void unet_correct<float>(Unet&, UnetAct&, const Lvl&, const float*, float*, float*, float*, double*,
                                  const RedBuf&, cudaStream_t);

}  // namespace gkb

// ---------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------

namespace {

template <class F>
int unet_guard(gkb_unet h, F&& fn) {
  if (!h) return GKB_ERR_INVALID_ARG;
  const gkb::CallBind call(h->u.stream);
  try {
    if (cudaSetDevice(h->device) != cudaSuccess) {
      (void)cudaGetLastError();
      return GKB_ERR_CUDA;
    }
    return fn();
  } catch (const gkb::Error& e) {
    h->last_error = e.msg;
    return e.code;
  } catch (const std::bad_alloc&) {
    h->last_error = "host allocation failed";
    return GKB_ERR_OOM;
  } catch (...) {
    h->last_error = "unexpected internal error";
    return GKB_ERR_CUDA;
  }
}

bool dev_ptr(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    (void)cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace

extern "C" {

int gkb_unet_create(gkb_unet* out, int c_in, int c1, int c2, int c_out, unsigned long long seed, void* stream) {
  if (!out) return GKB_ERR_INVALID_ARG;
  *out = nullptr;
  gkb_unet h = new (std::nothrow) gkb_unet_ctx();
  if (!h) return GKB_ERR_OOM;
  if (cudaGetDevice(&h->device) != cudaSuccess) {
    (void)cudaGetLastError();
    delete h;
    return GKB_ERR_CUDA;
  }
  h->u.stream = (cudaStream_t)stream;
  int rc = unet_guard(h, [&] {
    h->u.init(c_in, c1, c2, c_out, seed, (cudaStream_t)stream);
    gkb::check_cuda(cudaStreamSynchronize((cudaStream_t)stream), "init");
    return GKB_OK;
  });
  if (rc != GKB_OK) {
    delete h;
    return rc;
  }
  *out = h;
  return GKB_OK;
}

int gkb_unet_num_params(gkb_unet h, int64_t* n) {
  return unet_guard(h, [&] {
    if (!n) return GKB_ERR_INVALID_ARG;
    *n = h->u.nparams;
    return GKB_OK;
  });
}

int gkb_unet_get_params(gkb_unet h, float* params) {
  return unet_guard(h, [&] {
    if (!params) return GKB_ERR_INVALID_ARG;
    gkb::check_cuda(cudaMemcpyAsync(params, h->u.params.p, h->u.nparams * sizeof(float), cudaMemcpyDefault, h->u.stream), "copy");
    gkb::check_cuda(cudaStreamSynchronize(h->u.stream), "sync");
    return GKB_OK;
  });
}

int gkb_unet_set_params(gkb_unet h, const float* params) {
  return unet_guard(h, [&] {
    if (!params) return GKB_ERR_INVALID_ARG;
    gkb::check_cuda(cudaMemcpyAsync(h->u.params.p, params, h->u.nparams * sizeof(float), cudaMemcpyDefault, h->u.stream), "copy");
    gkb::check_cuda(cudaStreamSynchronize(h->u.stream), "sync");
    h->u.bf16_stale = true;
    return GKB_OK;
  });
}

int gkb_unet_forward(gkb_unet h, const float* x, int n, int hh, int w, float* y, int tensor_cores) {
  return unet_guard(h, [&] {
    if (!x || !y || !dev_ptr(x) || !dev_ptr(y)) throw gkb::Error{GKB_ERR_INVALID_ARG, "x and y must be device arrays"};
    const float* out = h->u.forward(h->u.act, x, n, hh, w, tensor_cores != 0, h->u.stream);
    gkb::check_cuda(cudaMemcpyAsync(y, out, (size_t)n * hh * w * h->u.c_out * sizeof(float), cudaMemcpyDeviceToDevice,
                                    h->u.stream), "copy");
    gkb::check_cuda(cudaStreamSynchronize(h->u.stream), "sync");
    return GKB_OK;
  });
}

int gkb_unet_loss_grad(gkb_unet h, const float* x, const float* target, int n, int hh, int w, double* loss, float* grad) {
  return unet_guard(h, [&] {
    if (!x || !target || !dev_ptr(x) || !dev_ptr(target)) throw gkb::Error{GKB_ERR_INVALID_ARG, "x and target must be device arrays"};
    const double l = h->u.loss_grad(x, target, n, hh, w);
    if (loss) *loss = l;
    if (grad) {
      gkb::check_cuda(cudaMemcpyAsync(grad, h->u.grads.p, h->u.nparams * sizeof(float), cudaMemcpyDefault, h->u.stream), "copy");
      gkb::check_cuda(cudaStreamSynchronize(h->u.stream), "sync");
    }
    return GKB_OK;
  });
}

int gkb_unet_adam_step(gkb_unet h, float lr, float beta1, float beta2, float eps) {
  return unet_guard(h, [&] {
    h->u.adam(lr, beta1, beta2, eps);
    gkb::check_cuda(cudaStreamSynchronize(h->u.stream), "sync");
    return GKB_OK;
  });
}

int gkb_unet_train(gkb_unet h, const float* x_img, const float* t_img, int64_t count, int hh, int w, int batch,
                   int steps, float lr, unsigned long long seed, double* losses) {
  return unet_guard(h, [&] {
    if (!x_img || !t_img || !dev_ptr(x_img) || !dev_ptr(t_img))
      throw gkb::Error{GKB_ERR_INVALID_ARG, "x_img and t_img must be device arrays"};
    h->u.ensure(h->u.act, batch < 1 ? 1 : batch, hh, w);
    h->u.train(x_img, t_img, count, hh, w, batch, steps, lr, seed, losses);
    return GKB_OK;
  });
}

int gkb_unet_set_target_scale(gkb_unet h, float s) {
  return unet_guard(h, [&] {
    if (!(s > 0) || !std::isfinite(s)) throw gkb::Error{GKB_ERR_INVALID_ARG, "target scale must be positive"};
    h->u.target_scale = s;
    return GKB_OK;
  });
}

int gkb_unet_get_target_scale(gkb_unet h, float* s) {
  return unet_guard(h, [&] {
    if (!s) return GKB_ERR_INVALID_ARG;
    *s = h->u.target_scale;
    return GKB_OK;
  });
}

const char* gkb_unet_last_error(gkb_unet h) { return h ? h->last_error.c_str() : "invalid handle"; }

int gkb_unet_destroy(gkb_unet h) {
  if (!h) return GKB_ERR_INVALID_ARG;
  cudaSetDevice(h->device);
  delete h;
  return GKB_OK;
}

}  // extern "C"
