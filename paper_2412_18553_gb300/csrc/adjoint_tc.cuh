// FP32-pair arithmetic and the per-triple values of the exact-slice epilogues
// (adjoint_tc.cu, frag.cu): W~, Y, R and 1/D at the positions of an orbit.
#pragma once
#include "fp_util.cuh"
#include "te_internal.h"

namespace te {

// value h + l; l a correction of about 2^-24 h, not always normalised
struct pr {
  float h, l;
};

__device__ __forceinline__ pr pr_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ pr pr_add(pr a, pr b) {
  const pr s = pr_two_sum(a.h, b.h);
  return {s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l))};
}
__device__ __forceinline__ pr pr_neg(pr a) { return {-a.h, -a.l}; }
__device__ __forceinline__ pr pr_sub(pr a, pr b) { return pr_add(a, pr_neg(b)); }
__device__ __forceinline__ pr pr_mul(pr a, pr b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = fmaf(a.h, b.h, -p);
  e = fmaf(a.h, b.l, e);
  e = fmaf(a.l, b.h, e);
  e = fmaf(a.l, b.l, e);
  return {p, e};
}
// s += a b
__device__ __forceinline__ void pr_fma(pr& s, pr a, pr b) { s = pr_add(s, pr_mul(a, b)); }
__device__ __forceinline__ pr pr_scale2(pr a, float k) { return {a.h * k, a.l * k}; }  // k a power of two
__device__ __forceinline__ float2 pr_norm2(pr a) {
  const float s = __fadd_rn(a.h, a.l);
  return make_float2(s, __fsub_rn(a.l, __fsub_rn(s, a.h)));
}
__device__ __forceinline__ pr pr_load(const float2* p) {
  const float2 x = __ldg(p);
  return {x.x, x.y};
}
__device__ __forceinline__ double pr_double(pr a) { return to_double(a.h) + to_double(a.l); }
// 1 / a: one correction of the FP32 reciprocal and its square
__device__ __forceinline__ pr pr_recip(pr a) {
  const float2 n = pr_norm2(a);
  const float r = __frcp_rn(n.x);
  float e = fmaf(-n.x, r, 1.f);
  e = fmaf(-n.y, r, e);
  return {r, fmaf(r * e, e, r * e)};
}
__device__ __forceinline__ pr pr_of(double x) {
  const float h = (float)x;
  return {h, (float)(x - (double)h)};
}

// x 2^-k as a pair, cut from the bits of x (x 2^-k below 2^-72 loses its low part)
__device__ __forceinline__ pr pr_bits(double x, int k) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint32_t sign = hi & 0x80000000u;
  const int E = (int)((hi >> 20) & 0x7FFu), fe = E - 1023 - k + 127;
  if (E == 0 || fe < 54) return {0.f, 0.f};
  if (fe > 254) return {__uint_as_float(sign | 0x7F800000u), 0.f};
  const float h = __uint_as_float(sign | ((uint32_t)fe << 23) | ((hi & 0xFFFFFu) << 3) | (lo >> 29));
  const float l = __uint2float_rn(lo & 0x1FFFFFFFu) * __uint_as_float((uint32_t)(fe - 52) << 23);
  return {h, __uint_as_float(__float_as_uint(l) | sign)};
}

// e with 2^e > m, from the high word of m (0 for zero)
__device__ __forceinline__ int exp_of_high(unsigned int hi) { return hi == 0u ? 0 : (int)((hi >> 20) & 0x7FFu) - 1022; }

// d 2^-shift in BF16 for an integer |d| <= 128: exact, so the upper half of
// the float is the value (the sum with 1.5 2^23 holds d in its low bits)
__device__ __forceinline__ uint32_t digit_bf16(int d, int shift) {
  const float f = __fsub_rn(__uint_as_float(0x4B400000u + (uint32_t)d), 12582912.0f);
  return __float_as_uint(__fmul_rn(f, __uint_as_float((uint32_t)(127 - shift) << 23))) >> 16;
}

// The epilogue's inputs as pairs.  ovs and t1 are relative to 2^(*e_ovs) and
// 2^(*e_t1).
struct PairInputs {
  int o, v;
  const pr* ovs;  // [o][v][o][v]  (ovov[i,a,j,b] + ovov[j,b,i,a]) / 2
  const pr* t1;   // [o][v]
  const pr *eps_o, *eps_v;
  const int *e_ovs, *e_t1;
};
struct PairBuffers {
  pr *ovs, *t1, *eps;
  unsigned int* hi;  // [0], [1]: high words of max |ovov|, |t1|; [2], [3]: their exponents (int)
};
inline PairInputs pair_inputs(const te_cluster* c, const PairBuffers& b, int o, int v) {
  (void)c;
  return PairInputs{o, v, b.ovs, b.t1, b.eps, b.eps + o, reinterpret_cast<const int*>(b.hi + 2),
                    reinterpret_cast<const int*>(b.hi + 3)};
}
cudaError_t launch_pair_inputs(const te_cluster* c, const PairBuffers& b, cudaStream_t s);

// Scale exponents of the slice sets a G block's segments read.
struct SliceExps {
  const int *e_ovvv, *e_t2, *e_t2L, *e_nooT;
};
// the contraction leaves G(p,q,r) relative to 2^(the largest scale of its segments)
__device__ __forceinline__ int g_exp(const SliceExps& x, int o, int p, int q, int r) {
  return max(max(x.e_ovvv[p] + x.e_t2[r * o + q], x.e_ovvv[q] + x.e_t2[r * o + p]),
             max(x.e_t2L[p] + x.e_nooT[q * o + r], x.e_t2L[q] + x.e_nooT[p * o + r]));
}

// W~ and Y of a triple are held relative to 2^E.
struct TripleScale {
  int E;
  float f[3], fy;  // factors of G_0, G_1, G_2 and of ovs t1
};
__device__ __forceinline__ TripleScale triple_scale(const PairInputs& in, const SliceExps& x, Triple T) {
  const int e0 = g_exp(x, in.o, T.i, T.j, T.k), e1 = g_exp(x, in.o, T.j, T.k, T.i), e2 = g_exp(x, in.o, T.k, T.i, T.j);
  const int ey = *in.e_ovs + *in.e_t1;
  TripleScale s;
  s.E = max(max(e0, e1), max(e2, ey));
  s.f[0] = ldexpf(1.f, e0 - s.E);
  s.f[1] = ldexpf(1.f, e1 - s.E);
  s.f[2] = ldexpf(1.f, e2 - s.E);
  s.fy = ldexpf(1.f, ey - s.E);
  return s;
}
__device__ __forceinline__ pr occ_energy(const PairInputs& in, Triple T) {
  return pr_add(pr_add(in.eps_o[T.i], in.eps_o[T.j]), in.eps_o[T.k]);
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

// Positions abc, acb, bac, bca, cab, cba.  G_g at the six permutations of
// (a, b, c) is read once; W~ at position n is G_0 there, G_1 at the cyclic
// successor and G_2 at the one after.
__device__ __forceinline__ void orbit_w(const float2* G, int64_t v, const TripleScale& s, int a, int b, int c, pr* W) {
  const int64_t v2 = v * v, v3 = v2 * v;
  const int64_t at[6] = {a * v2 + b * v + c, a * v2 + c * v + b, b * v2 + a * v + c,
                         b * v2 + c * v + a, c * v2 + a * v + b, c * v2 + b * v + a};
  constexpr int r1[6] = {3, 5, 1, 4, 0, 2}, r2[6] = {4, 2, 5, 0, 3, 1};
#pragma unroll
  for (int n = 0; n < 6; ++n)
    W[n] = pr_add(pr_add(pr_scale2(pr_load(G + at[n]), s.f[0]), pr_scale2(pr_load(G + v3 + at[r1[n]]), s.f[1])),
                  pr_scale2(pr_load(G + 2 * v3 + at[r2[n]]), s.f[2]));
}
// Y = ovs(i,x,j,y) t1(k,z) + ovs(j,y,k,z) t1(i,x) + ovs(i,x,k,z) t1(j,y)
__device__ __forceinline__ void orbit_y(const PairInputs& in, Triple T, const TripleScale& s, int a, int b, int c,
                                        pr* Y) {
  const int64_t v = in.v, o = in.o;
  const int p[6][3] = {{a, b, c}, {a, c, b}, {b, a, c}, {b, c, a}, {c, a, b}, {c, b, a}};
  auto ovs = [&](int p1, int x, int p2, int y) { return in.ovs[((p1 * v + x) * o + p2) * v + y]; };
#pragma unroll
  for (int n = 0; n < 6; ++n) {
    const int x = p[n][0], y = p[n][1], z = p[n][2];
    pr t = pr_mul(ovs(T.i, x, T.j, y), in.t1[(int64_t)T.k * v + z]);
    pr_fma(t, ovs(T.j, y, T.k, z), in.t1[(int64_t)T.i * v + x]);
    pr_fma(t, ovs(T.i, x, T.k, z), in.t1[(int64_t)T.j * v + y]);
    Y[n] = pr_scale2(t, s.fy);
  }
}
// R at every position (identity 4, 3-cycles +1, transpositions -2): 3 x_p +
// (sum over p's parity class) - 2 (sum over the other class)
__device__ __forceinline__ void r_orbit_pairs(const pr* x, pr* r) {
  const pr se = pr_add(pr_add(x[0], x[3]), x[4]), so = pr_add(pr_add(x[1], x[2]), x[5]);
  const pr ue = pr_sub(se, pr_scale2(so, 2.f)), uo = pr_sub(so, pr_scale2(se, 2.f));
#pragma unroll
  for (int n = 0; n < 6; ++n) {
    const bool even = n == 0 || n == 3 || n == 4;
    r[n] = pr_add(pr_add(pr_scale2(x[n], 2.f), x[n]), even ? ue : uo);
  }
}

}  // namespace te
