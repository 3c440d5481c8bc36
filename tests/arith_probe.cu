// Counts the values on which the framework's own arithmetic differs in a bit
// from CUDA's: div_by against the division, to_f64 against the conversion.
#include <stdint.h>

#include "common.cuh"

namespace {

__device__ uint64_t mix(uint64_t x) {  // splitmix64
  x += 0x9e3779b97f4a7c15ull;
  x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
  x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
  return x ^ (x >> 31);
}
__device__ double bits(uint64_t u) { return __longlong_as_double((long long)u); }
// significand f (52 bits) at biased exponent e
__device__ double make(uint64_t f, unsigned e) { return bits((f & 0xfffffffffffffull) | ((uint64_t)(e & 0x7ff) << 52)); }
__device__ bool same(double a, double b) {
  return __double_as_longlong(a) == __double_as_longlong(b) || (a != a && b != b);
}

// kind 0: any pair of bit patterns; 1: exponents near 1; 2: every pair of
// significands of 10 bits; 3: dividends next to b times a number halfway
// between two doubles
__global__ void k_div(int kind, long long n, unsigned long long* bad) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const uint64_t u = mix(2 * t), v = mix(2 * t + 1);
  double a, b;
  if (kind == 0) {
    a = bits(u);
    b = bits(v);
  } else if (kind == 1) {
    a = make(u, 1023 - 32 + (u >> 58));
    b = make(v, 1023 - 32 + (v >> 58));
  } else if (kind == 2) {
    a = make((uint64_t)(t & 1023) << 42, 1023);
    b = make((uint64_t)((t >> 10) & 1023) << 42, 1023);
  } else {
    b = make(u | 1, 1023);
    const double q = make(v, 1022 + (v >> 63));
    const double half = 0.5 * (make(v + 1, 1022 + (v >> 63)) - q);  // half an ulp of q
    a = fma(b, q, b * half);
    a = bits((uint64_t)__double_as_longlong(a) + (v >> 60 & 3) - 1);  // and its neighbours
  }
  if (!same(gkb::div_by(a, b, 1.0 / b), a / b)) atomicAdd(bad, 1ull);
}

// groups of four floats: every bit pattern in turn beside three hashed ones
// (mixed: of any kind, else normal)
__global__ void k_cvt(int mixed, unsigned long long* bad) {
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;  // 2^22 threads of 1024 patterns
  for (unsigned k = 0; k < 1024; ++k) {
    const unsigned p = t * 1024u + k;
    const uint64_t h = mix(p);
    float v[4] = {__uint_as_float(p), __uint_as_float((unsigned)h), __uint_as_float((unsigned)(h >> 32)), 1.f};
    if (!mixed) {
      v[1] = 1.5f;
      v[2] = -3e-38f;
    }
    double z[4];
    gkb::to_f64(v, z);
    for (int q = 0; q < 4; ++q)
      if (!same(z[q], (double)v[q])) atomicAdd(bad, 1ull);
  }
}

}  // namespace

// -1: a CUDA error
extern "C" long long probe(int what, int kind, long long n) {
  unsigned long long* bad = nullptr;
  unsigned long long host = 0;
  if (cudaMalloc(&bad, sizeof host) != cudaSuccess) return -1;
  cudaMemset(bad, 0, sizeof host);
  if (what == 0) k_div<<<(unsigned)((n + 255) / 256), 256>>>(kind, n, bad);
  else k_cvt<<<(1u << 22) / 256, 256>>>(kind, bad);
  const cudaError_t e = cudaMemcpy(&host, bad, sizeof host, cudaMemcpyDeviceToHost);
  cudaFree(bad);
  return e == cudaSuccess ? (long long)host : -1;
}
