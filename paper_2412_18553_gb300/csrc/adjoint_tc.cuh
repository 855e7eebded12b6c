// Shared by the exact-slice adjoint and projected energy (adjoint_tc.cu, frag.cu):
// slice digits, the scales of their G blocks, and the order in which the
// epilogues take the orbits.
#pragma once
#include "fp_util.cuh"
#include "te_internal.h"

namespace te {

// e with 2^e > m, from the high word of m (0 for zero)
__device__ __forceinline__ int exp_of_high(unsigned int hi) { return hi == 0u ? 0 : (int)((hi >> 20) & 0x7FFu) - 1022; }

// d 2^-shift in BF16 for an integer |d| <= 128: exact, so the upper half of
// the float is the value (the sum with 1.5 2^23 holds d in its low bits)
__device__ __forceinline__ uint32_t digit_bf16(int d, int shift) {
  const float f = __fsub_rn(__uint_as_float(0x4B400000u + (uint32_t)d), 12582912.0f);
  return __float_as_uint(__fmul_rn(f, __uint_as_float((uint32_t)(127 - shift) << 23))) >> 16;
}

// Scale exponents of the slice sets a G block's segments read.
struct SliceExps {
  const int *e_ovvv, *e_t2, *e_t2L, *e_nooT;
};
// the contraction leaves G(p,q,r) relative to 2^(the largest scale of its segments)
__device__ __forceinline__ int g_exp(const SliceExps& x, int o, int p, int q, int r) {
  return max(max(x.e_ovvv[p] + x.e_t2[r * o + q], x.e_ovvv[q] + x.e_t2[r * o + p]),
             max(x.e_t2L[p] + x.e_nooT[q * o + r], x.e_t2L[q] + x.e_nooT[p * o + r]));
}

// orbit index t = a(a+1)(a+2)/6 + b(b+1)/2 + c -> (a, b, c), a >= b >= c
// (FP32 estimates, exact integer fix-ups)
__device__ __forceinline__ void orbit_abc(int64_t t, int* pa, int* pb, int* pc) {
  int a = (int)cbrtf(6.0f * (float)t);
  while (a > 0 && (int64_t)a * (a + 1) * (a + 2) / 6 > t) --a;
  while ((int64_t)(a + 1) * (a + 2) * (a + 3) / 6 <= t) ++a;
  const int64_t rem = t - (int64_t)a * (a + 1) * (a + 2) / 6;
  int b = (int)sqrtf(2.0f * (float)rem);
  while (b > 0 && (int64_t)b * (b + 1) / 2 > rem) --b;
  while ((int64_t)(b + 1) * (b + 2) / 2 <= rem) ++b;
  *pa = a;
  *pb = b;
  *pc = (int)(rem - (int64_t)b * (b + 1) / 2);
}

// The epilogues' orbits go by block triples of 8 x 8 x 8 (X >= Y >= Z), half of one
// per block of 256 threads and step.  A warp covers 2 x 4 x 4 of (a, b, c), so
// that of the six positions' accesses (8 bytes each, contiguous in the last
// index) those ending in b or c use whole 32-byte sectors and those ending in a
// half of them; 32 consecutive c used a quarter in four positions of six.
struct OrbitTile {
  int la, lb, lc;
};
__device__ __forceinline__ OrbitTile orbit_tile() {
  const int t = threadIdx.x;
  return {((t >> 4) & 1) | ((t >> 6) & 2), ((t >> 2) & 3) | ((t >> 4) & 4), (t & 3) | ((t >> 3) & 4)};
}
__device__ __forceinline__ int64_t orbit_steps(int v) {
  const int64_t nb = (v + 7) / 8;
  return nb * (nb + 1) * (nb + 2) / 3;  // two per block triple
}
// this thread's orbit in step t; false where it is none (a >= b >= c, a < v)
__device__ __forceinline__ bool orbit_at(const OrbitTile& o, int64_t t, int v, int* a, int* b, int* c) {
  int X, Y, Z;
  orbit_abc(t >> 1, &X, &Y, &Z);
  *a = X * 8 + (int)(t & 1) * 4 + o.la;
  *b = Y * 8 + o.lb;
  *c = Z * 8 + o.lc;
  return *a < v && *a >= *b && *b >= *c;
}

}  // namespace te
