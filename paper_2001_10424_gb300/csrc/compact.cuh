// compact.cuh - the compact ordering of include/gkb.h, and operator products
// that read and write it directly.
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"

namespace gkb {

struct Compact {
  int dim;
  int lo[3][3];    // low corner of the active box of component c
  int ext[3][3];   // extents of that box
  long long base[3];
  long long m;
};

inline Compact make_compact(const Lvl& L) {
  Compact c{};
  c.dim = L.dim;
  long long off = 0;
  for (int comp = 0; comp < L.dim; ++comp) {
    for (int a = 0; a < 3; ++a) {
      if (a >= L.dim) { c.lo[comp][a] = 0; c.ext[comp][a] = 1; continue; }
      if (a == comp) {
        const int lo = L.nat[2 * a] ? 0 : 1;
        const int hi = L.nat[2 * a + 1] ? L.n[a] : L.n[a] - 1;
        c.lo[comp][a] = lo;
        c.ext[comp][a] = hi - lo + 1;
      } else {
        c.lo[comp][a] = 0;
        c.ext[comp][a] = L.n[a];
      }
    }
    c.base[comp] = off;
    off += (long long)c.ext[comp][0] * c.ext[comp][1] * c.ext[comp][2];
  }
  c.m = off;
  return c;
}

// y = op(x) (GKB_OP_*) on compact device vectors that do not overlap, for a
// constant-viscosity level with N = n I: one launch on s
void apply_compact(const Lvl& L, int op, const double* x, double* y, cudaStream_t s);

// the two device ranges share memory
inline bool overlap(const double* x, long long nx, const double* y, long long ny) {
  return x < y + ny && y < x + nx;
}

}  // namespace gkb
