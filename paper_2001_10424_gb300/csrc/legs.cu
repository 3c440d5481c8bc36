// legs.cu - launches of the fused V-cycle legs (legs.cuh).
#include <climits>
#include "legs.cuh"
#include "solver.cuh"

namespace gkb {

template <typename T, int DEG, int KIND, bool DOWN>
__global__ void __launch_bounds__(LegShape<DEG, KIND, DOWN>::NT, KIND == LEG_8 ? 1 : 2)
    k_leg(const __grid_constant__ LegArgs<T> A) {
  extern __shared__ __align__(16) unsigned char leg_sm[];
  leg_body<T, DEG, KIND, DOWN>(native_blk(), A, (T*)leg_sm);
}

namespace {

template <typename T, int DEG, int KIND, bool DOWN>
void launch_leg(const LegArgs<T>& A, cudaStream_t s) {
  using G = LegShape<DEG, KIND, DOWN>;
  constexpr size_t sm = G::template smem<T>();
  if (sm > 48 * 1024)
    GKB_CUDA(cudaFuncSetAttribute(k_leg<T, DEG, KIND, DOWN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  k_leg<T, DEG, KIND, DOWN><<<G::grid(A.L), G::NT, sm, s>>>(A);
  GKB_CUDA(cudaGetLastError());
}

template <typename T, int DEG, bool DOWN>
void launch_kind(int kind, const LegArgs<T>& A, cudaStream_t s) {
  if constexpr (sizeof(T) == 4) {
    if (kind == LEG_STRIP) return launch_leg<T, DEG, LEG_STRIP, DOWN>(A, s);
    if (kind == LEG_VAR) return launch_leg<T, DEG, LEG_VAR, DOWN>(A, s);
  }
  launch_leg<T, DEG, LEG_8, DOWN>(A, s);
}

template <typename T, bool DOWN>
void launch_degree(int degree, int kind, const LegArgs<T>& A, cudaStream_t s) {
  if (degree == 1) launch_kind<T, 1, DOWN>(kind, A, s);
  else if (degree == 2) launch_kind<T, 2, DOWN>(kind, A, s);
  else launch_kind<T, 3, DOWN>(kind, A, s);
}

// Which levels run as legs. FP64: the halo's recomputation costs FP64-pipe
// time (three times a tile's own work for 8 x 8 cells), which pays only while
// a separate launch is mostly latency, up to 128^2 (V-cycle share of a 128^2
// level 165 -> 72 us; with 256^2 as legs too, a 256^2 solve gains 6 % but two
// concurrent 1024^2 solves lose 2 %). FP32: everywhere; strips above 64^2
// (256^2 solve 27.1 ms, with 8 x 8 tiles 26.5 ms; 1024^2 62 against 94 ms).
template <typename T>
int leg_kind(const Lvl& L) {
  const long long cells = (long long)L.n[0] * L.n[1];
  if (sizeof(T) == 8) return cells <= 128 * 128 ? LEG_8 : LEG_OFF;
  return cells <= 64 * 64 ? LEG_8 : LEG_STRIP;
}

}  // namespace

template <typename T>
void gmg_leg_args(const Gmg<T>& G, int l, const T* b, const T* rd, T* z0, LegArgs<T>& A) {
  const auto& V = G.lev[l];
  const auto& C = G.lev[l + 1];
  A = LegArgs<T>{};
  A.L = V.L;
  A.Lc = C.L;
  A.b = b;
  A.rd = rd;
  A.bfull = V.d.p;
  A.xpre = V.r.p;
  A.xc = C.x.p;
  A.xout = l == 0 ? z0 : V.x.p;
  A.bc = C.b.p;
  A.tmp = C.x.p;
  A.table = V.table.p;
  for (int k = 0; k < G.degree; ++k) {
    A.ca[k] = (T)V.ca[k];
    A.cb[k] = (T)V.cb[k];
    if (!V.fold_in.empty()) A.fs[k] = fold2_scaled<T>(V.fold_in.data(), (double)(T)V.ca[k]);
  }
}
template void gmg_leg_args<float>(const Gmg<float>&, int, const float*, const float*, float*, LegArgs<float>&);
template void gmg_leg_args<double>(const Gmg<double>&, int, const double*, const double*, double*, LegArgs<double>&);

template <typename T>
void gmg_leg_plan(Gmg<T>& G) {
  for (size_t l = 0; l < G.lev.size(); ++l) {
    auto& V = G.lev[l];
    V.leg = LEG_OFF;
    if (l + 1 == G.lev.size() || V.L.dim != 2 || !V.L.fast || G.degree > LEG_MAX_DEG) continue;
    if (V.L.nvel > INT_MAX) continue;  // the legs index with 32 bits
    if (!V.fold_in.empty() && cheb2_level(V.L)) V.leg = leg_kind<T>(V.L);
    // FP32 variable viscosity with N = n I and the Laplacian form
    else if (sizeof(T) == 4 && V.L.mu32 && !V.L.nw32 && !V.L.sym) V.leg = LEG_VAR;
  }
}
template void gmg_leg_plan<float>(Gmg<float>&);
template void gmg_leg_plan<double>(Gmg<double>&);

template <typename T>
void gmg_leg(const Gmg<T>& G, int l, bool down, const T* b, const T* rd, T* z0, cudaStream_t s) {
  LegArgs<T> A;
  gmg_leg_args<T>(G, l, b, rd, z0, A);
  ProfScope ps_(GKB_KC_SMOOTH, s, lvl_unknowns(A.L));
  if (down) launch_degree<T, true>(G.degree, G.lev[l].leg, A, s);
  else launch_degree<T, false>(G.degree, G.lev[l].leg, A, s);
}
template void gmg_leg<float>(const Gmg<float>&, int, bool, const float*, const float*, float*, cudaStream_t);
template void gmg_leg<double>(const Gmg<double>&, int, bool, const double*, const double*, double*, cudaStream_t);

}  // namespace gkb
