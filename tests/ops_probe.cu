// Operator products of one 2D level through the launchers that the solver
// uses (Ops<T>), on padded arrays: the product alone, the same with the
// deep-interior fast paths off, and the product with its inner product. Counts
// the values in which the latter two differ in a bit from the first.
#include <string.h>

#include <cmath>
#include <limits>
#include <vector>

#include "solver.cuh"

namespace {

using namespace gkb;

double hashed(unsigned long long t) {  // in [-1, 1)
  t += 0x9e3779b97f4a7c15ull;
  t = (t ^ (t >> 30)) * 0xbf58476d1ce4e5b9ull;
  t = (t ^ (t >> 27)) * 0x94d049bb133111ebull;
  t ^= t >> 31;
  return (double)(t >> 11) * 0x1p-52 - 1.0;
}

template <typename T>
std::vector<T> host(const DevBuf<T>& b) {
  std::vector<T> v(b.n);
  GKB_CUDA(cudaMemcpy(v.data(), b.p, b.n * sizeof(T), cudaMemcpyDeviceToHost));
  return v;
}
template <typename T>
void put(DevBuf<T>& b, const std::vector<T>& v) {
  b.alloc(v.size());
  GKB_CUDA(cudaMemcpy(b.p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice));
}
template <typename T>
long long differing(const std::vector<T>& a, const std::vector<T>& b) {
  long long k = 0;
  for (size_t t = 0; t < a.size(); ++t) k += memcmp(&a[t], &b[t], sizeof(T)) != 0;
  return k;
}

void set_mu(Lvl& L, const float* m) { L.mu32 = m; }
void set_mu(Lvl&, const double*) {}

template <typename T>
void run(const int* n, const int* nat, int var, int mode, long long* diff, double* dot) {
  Lvl L = make_level(2, n, 1.0 / n[0], nat, 300.0);
  L.mu0 = var ? 1.0 : 1.3;
  finish_level(L);
  // the active faces
  std::vector<double> ones((size_t)L.nvel, 1.0);
  DevBuf<double> compact, mask;
  put(compact, ones);
  mask.alloc(L.nvel);
  pack_velocity(L, compact.p, mask.p, 0);
  const std::vector<double> on = host(mask);
  std::vector<T> x(L.nvel), bad(L.nvel), mu(L.ncell, (T)0);
  for (long long t = 0; t < L.nvel; ++t) {
    x[t] = on[t] != 0 ? (T)hashed(t) : (T)0;
    bad[t] = on[t] != 0 ? std::numeric_limits<T>::quiet_NaN() : (T)0;
  }
  for (int j = 0; j < n[1]; ++j)
    for (int i = 0; i < n[0]; ++i) mu[(long long)j * L.P + i] = (T)exp(0.7 * hashed(77777777 + (long long)j * n[0] + i));
  DevBuf<T> xd, md, y[3];
  put(xd, x);
  put(md, mu);
  if (var) set_mu(L, md.p);
  for (auto& b : y) put(b, bad);
  DevBuf<double> partial, out;
  DevBuf<unsigned> ticket;
  partial.alloc(Ops<T>::face_blocks(L) * 4 + 64);
  ticket.alloc(1);
  out.alloc(4);
  const RedBuf red{partial.p, ticket.p};
  Lvl G = L;
  G.fast = 0;
  Ops<T>::apply(L, mode, xd.p, y[0].p, 0);
  Ops<T>::apply(G, mode, xd.p, y[1].p, 0);
  Ops<T>::apply_dot(L, mode, xd.p, y[2].p, red, FIN_STORE, out.p, 0);
  GKB_CUDA(cudaDeviceSynchronize());
  GKB_CUDA(cudaGetLastError());
  const std::vector<T> a = host(y[0]);
  diff[0] = differing(a, host(y[1]));
  diff[1] = differing(a, host(y[2]));
  double s = 0.0, abs = 0.0;
  for (long long t = 0; t < L.nvel; ++t) {
    s += (double)x[t] * (double)a[t];
    abs += fabs((double)x[t] * (double)a[t]);
  }
  *dot = fabs(host(out)[0] - s) / abs;
}

}  // namespace

// diff: values that differ with the fast paths off, and in the product with
// its inner product; dot: that inner product's error over the sum of the
// absolute products. Returns 0, or the library's error code.
extern "C" int probe(int fp64, const int* n, const int* nat, int var, int mode, long long* diff, double* dot) {
  try {
    if (fp64) run<double>(n, nat, var, mode, diff, dot);
    else run<float>(n, nat, var, mode, diff, dot);
    return 0;
  } catch (const Error& e) {
    return e.code;
  }
}
