// Fragment-projected E(T) (Eq. E_corr_CCSD_T with a general C^f) on the
// strided-view contractions of the adjoint; see the comment below.
#include <cuda_bf16.h>

#include <algorithm>
#include <new>
#include <vector>

#include "adjoint_tc.cuh"
#include "fp_util.cuh"
#include "strided.h"
#include "tc_path.h"
#include "view_tc.h"
#include "te_internal.h"

namespace te {

te_status ensure_triples_public(Handle* h, int nocc);

// ---------------------------------------------------------------------------
// Fragment-projected E(T): Eq. E_corr_CCSD_T with a general C^f
// ---------------------------------------------------------------------------
// E_x = (1/3) sum_{ijk} sum_{abc} sum_{i'} C_{ii'} W~_{i'jk} R[Z]_{ijk}: C acts on
// the first occupied index of W~.  Summed over all ordered triples, C on any
// one of the three occupied indices gives the same total, so every unique
// triple takes the average S W~ = 1/3 (C_1 + C_2 + C_3) W~, which keeps the
// joint (ijk, abc) permutation symmetry of W~:
//   share_{ijk} = (m/3) sum_{abc} (S W~)_{ijk} R[V]_{ijk} / D_{ijk},  V = W~ + Y.
// S W~ = P[S X] groups into G-like blocks like W~ = P[X].  C on one occupied
// index of a G segment lands on exactly one of its two factors, and summing
// the three placements gives two products per segment:
//   SG(p,q,r) = 1/3 [ ovvvC[p] t2[r,q] + ovvv[p] t2C[r,q] + ovvvC[q] t2[r,p] + ovvv[q] t2C[r,p]
//                     + t2LC[p] nooT[q][r] + t2L[p] nooTC[q][r] + t2LC[q] nooT[p][r] + t2L[q] nooTC[p][r] ]
// with ovvvC = C on the first index of ovvv; t2C = C on the first plus C on
// the second index of t2; t2LC = the t2L copy of t2 with C on its second
// index; nooTC = the nooT copy of ooov with C on its first plus on its third
// index.

// out[a][p][b] (+)= sum_{p'} C[p][p'] in[a][p'][b]: C on one occupied index,
// `outer` and `inner` the sizes around it; fixed summation order
__global__ void k_occ_transform(const double* __restrict__ in, const double* __restrict__ C, int o, int64_t outer,
                                int64_t inner, double* __restrict__ out, int accumulate) {
  const int64_t n = outer * o * inner;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t a = e / (o * inner), b = e % inner;
    const int p = (int)((e / inner) % o);
    const double* src = in + a * o * inner + b;
    double s = 0.0;
    for (int q = 0; q < o; ++q) s += C[p * o + q] * src[q * inner];
    out[e] = accumulate ? out[e] + s : s;
  }
}

// per-block sums of (S W~) R[V] / D over the abc of one triple, one thread per
// orbit representative a >= b >= c
__global__ void __launch_bounds__(256) k_energy_proj(AdjArgs A, const double* __restrict__ SG) {
  __shared__ double red[8];
  const int64_t v = A.v, v3 = v * v * v;
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  double contrib = 0.0;
  if (e < v3) {
    const int a = (int)(e / (v * v)), b = (int)((e / v) % v), c = (int)(e % v);
    if (a >= b && b >= c) {
      double W[6], Y[6], V[6], RV[6];
      orbit_values(A, a, b, c, W, Y);
#pragma unroll
      for (int n = 0; n < 6; ++n) V[n] = W[n] + Y[n];
      r_orbit(V, RV);
      AdjArgs S = A;
      S.G = SG;
      const int p[6][3] = {{a, b, c}, {a, c, b}, {b, a, c}, {b, c, a}, {c, a, b}, {c, b, a}};
      const unsigned distinct = orbit_distinct(a, b, c);
      const double D = (A.eps_o[A.i] + A.eps_o[A.j] + A.eps_o[A.k]) - A.eps_v[a] - A.eps_v[b] - A.eps_v[c];
      double t = 0.0;
#pragma unroll
      for (int n = 0; n < 6; ++n)
        if (distinct >> n & 1u) t += wt_at(S, p[n][0], p[n][1], p[n][2]) * RV[n];
      contrib = t / D;
    }
  }
  for (int off = 16; off > 0; off >>= 1) contrib += __shfl_down_sync(0xffffffffu, contrib, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = contrib;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += red[w];
    A.epart[blockIdx.x] = t;
  }
}

// ---------------------------------------------------------------------------
// float64 form
// ---------------------------------------------------------------------------

struct FragWork {
  double *ovvvC, *t2C, *t2C2, *ooovC;      // C on occupied indices of the inputs
  double *t2L, *nooT, *ovs;                // float64 helper copies of the inputs
  double *t2LC, *nooTC, *ovs_unused;       // the same of t2C2 and ooovC
  double *G, *SG;                          // [3][v][v][v] each
  double *epart, *shares, *scratch;
  int64_t scratch_cap;
};

namespace {

struct Carve {
  char* base;
  size_t off = 0;
  char* take(size_t bytes) {
    off = (off + 1023) & ~size_t(1023);
    char* r = base ? base + off : nullptr;
    off += bytes;
    return r;
  }
  double* d(int64_t n) { return reinterpret_cast<double*>(take((size_t)n * 8)); }
};

// carve the workspace (base = nullptr: sizes only)
size_t frag_layout(int64_t o, int64_t v, char* base, FragWork* W) {
  const int64_t v3 = v * v * v, nt = num_unique_triples(o), nblk = (v3 + 255) / 256;
  Carve c{base};
  W->ovvvC = c.d(o * v3);
  W->t2C = c.d(o * o * v * v);
  W->t2C2 = c.d(o * o * v * v);
  W->ooovC = c.d(o * o * o * v);
  W->t2L = c.d(o * v * v * o);
  W->nooT = c.d(o * o * v * o);
  W->ovs = c.d(o * v * o * v);
  W->t2LC = c.d(o * v * v * o);
  W->nooTC = c.d(o * o * v * o);
  W->ovs_unused = c.d(o * v * o * v);
  W->G = c.d(3 * v3);
  W->SG = c.d(3 * v3);
  W->epart = c.d(nblk);
  W->shares = c.d(std::max<int64_t>(1, nt));
  W->scratch_cap = splitk_cap(o, v);
  W->scratch = c.d(W->scratch_cap);
  return c.off + 1024;
}

// C on the occupied indices of the inputs
cudaError_t transform_inputs(Handle* h, const te_cluster* c, const double* cf, double* ovvvC, double* t2C, double* t2C2,
                             double* ooovC, cudaStream_t s) {
  const int o = (int)c->nocc, v = (int)c->nvir;
  const int64_t v2 = (int64_t)v * v, v3 = v2 * v;
  auto tr = [&](const double* in, int64_t outer, int64_t inner, double* out, int acc) {
    const int64_t n = outer * o * inner;
    k_occ_transform<<<(unsigned)std::min<int64_t>((n + 255) / 256, 8 * 1024), 256, 0, s>>>(in, cf, o, outer,
                                                                                           inner, out, acc);
    ++h->n_launches;
  };
  tr(c->ovvv, 1, v3, ovvvC, 0);                           // ovvv[p,a,b,d]: first index
  tr(c->t2, 1, (int64_t)o * v2, t2C, 0);                  // t2[r,q,a,b]: first index
  tr(c->t2, o, v2, t2C, 1);                               //   plus second index
  tr(c->t2, o, v2, t2C2, 0);                              // second index only
  tr(c->ooov, 1, (int64_t)o * o * v, ooovC, 0);           // ooov[p,l,r,z]: first index
  tr(c->ooov, (int64_t)o * o, v, ooovC, 1);               //   plus third index
  return cudaGetLastError();
}

te_status run_frag_fp64(Handle* h, const te_cluster* c, const double* cf, const FragWork& W, cudaStream_t s) {
  const int o = (int)c->nocc, v = (int)c->nvir;
  const int64_t v2 = (int64_t)v * v, v3 = v2 * v, nt = num_unique_triples(o), nblk = (v3 + 255) / 256;
  cudaError_t e = transform_inputs(h, c, cf, W.ovvvC, W.t2C, W.t2C2, W.ooovC, s);
  if (e != cudaSuccess) return fail(TE_ECUDA, "transform launch: %s", cudaGetErrorString(e));
  // float64 helper copies: t2L, nooT, ovs of the inputs; t2L of t2C2, nooT of ooovC
  Prepared P{};
  P.o = o; P.v = v; P.eps_o = c->eps_o; P.eps_v = c->eps_v; P.ovvv = c->ovvv; P.t2 = c->t2; P.t1 = c->t1;
  P.t2L = W.t2L; P.nooT = W.nooT; P.ovs = W.ovs;
  e = launch_prep_fp64(c, &P, s);
  te_cluster cx = *c;
  cx.t2 = W.t2C2;
  cx.ooov = W.ooovC;
  Prepared PX{};
  PX.o = o; PX.v = v; PX.t2L = W.t2LC; PX.nooT = W.nooTC; PX.ovs = W.ovs_unused;
  if (e == cudaSuccess) e = launch_prep_fp64(&cx, &PX, s);
  h->n_launches += 6;
  if (e != cudaSuccess) return fail(TE_ECUDA, "prep: %s", cudaGetErrorString(e));
  std::vector<Triple> trip = unique_triples(o);
  const double third = 1.0 / 3.0;
  for (int64_t t = 0; t < nt && e == cudaSuccess; ++t) {
    const Triple T = trip[t];
    e = cudaMemsetAsync(W.SG, 0, sizeof(double) * 3 * v3, s);
    if (e != cudaSuccess) break;
    e = launch_gemm_fp64(&P, h->d_triples, t, 1, W.G, h->num_sms, s);
    ++h->n_launches;
    for (int gi = 0; gi < 3 && e == cudaSuccess; ++gi) {
      int pp, qq, rr;
      if (gi == 0) { pp = T.i; qq = T.j; rr = T.k; }
      else if (gi == 1) { pp = T.j; qq = T.k; rr = T.i; }
      else { pp = T.k; qq = T.i; rr = T.j; }
      double* SGg = W.SG + gi * v3;
      // float64: the eight products of SG(p,q,r), rows (x, y), columns z
      auto run = [&](const double* A, int64_t am1, int64_t am2, int64_t K, const double* B, int64_t bn) {
        if (e == cudaSuccess)
          e = gemm_strided(GemmView{A, B, SGg, v, v, v, K, 1, am1, am2, 1, 0, 1, 0, bn, v2, v, 1, third}, h->num_sms,
                           W.scratch, W.scratch_cap, s, &h->n_launches);
      };
      const int64_t orq = ((int64_t)rr * o + qq) * v2, orp = ((int64_t)rr * o + pp) * v2;
      run(W.ovvvC + pp * v3, v2, v, v, c->t2 + orq, v);     // S1: ovvvC[p,x,y,d] t2[r,q,z,d]
      run(c->ovvv + pp * v3, v2, v, v, W.t2C + orq, v);     //     ovvv[p] t2C[r,q]
      run(W.ovvvC + qq * v3, v, v2, v, c->t2 + orp, v);     // S2: ovvvC[q,y,x,d] t2[r,p,z,d]
      run(c->ovvv + qq * v3, v, v2, v, W.t2C + orp, v);     //     ovvv[q] t2C[r,p]
      const int64_t lp = (int64_t)pp * v2 * o, lq = (int64_t)qq * v2 * o;
      const int64_t nqr = ((int64_t)qq * o + rr) * v * o, npr = ((int64_t)pp * o + rr) * v * o;
      run(W.t2LC + lp, o, (int64_t)v * o, o, W.nooT + nqr, o);   // S3: t2LC[p][y][x][l] nooT[q][r][z][l]
      run(W.t2L + lp, o, (int64_t)v * o, o, W.nooTC + nqr, o);   //     t2L[p] nooTC[q][r]
      run(W.t2LC + lq, (int64_t)v * o, o, o, W.nooT + npr, o);   // S4: t2LC[q][x][y][l] nooT[p][r][z][l]
      run(W.t2L + lq, (int64_t)v * o, o, o, W.nooTC + npr, o);   //     t2L[q] nooTC[p][r]
    }
    if (e != cudaSuccess) break;
    AdjArgs A{};
    A.o = o; A.v = v; A.i = T.i; A.j = T.j; A.k = T.k;
    A.G = W.G; A.ovs = W.ovs; A.t1 = c->t1; A.eps_o = c->eps_o; A.eps_v = c->eps_v; A.epart = W.epart;
    k_energy_proj<<<(unsigned)nblk, 256, 0, s>>>(A, W.SG);
    e = launch_sum_share(W.epart, nblk, (double)T.m / 3.0, W.shares + t, s);
    h->n_launches += 2;
  }
  if (e != cudaSuccess) return fail(TE_ECUDA, "projected energy launch: %s", cudaGetErrorString(e));
  return TE_OK;
}

// ---------------------------------------------------------------------------
// exact-slice form: batches of triples
// ---------------------------------------------------------------------------

constexpr int FRAG_MAX_BATCH = 8;
constexpr int64_t FRAG_BATCH_BYTES = int64_t(1) << 30;  // G and SG of a batch

struct FragOz {
  double *ovvvC, *t2C, *t2C2, *ooovC, *ovs;
  float2 *G, *SG;  // [slot][3][v^3]
  int64_t stride;  // float2 between the slots of each
  double *epart, *shares;
  char* slices[3];
};

int frag_batch(int64_t o, int64_t v) {
  return (int)std::max<int64_t>(1, std::min<int64_t>({FRAG_MAX_BATCH, FRAG_BATCH_BYTES / (48 * v * v * v),
                                                      std::max<int64_t>(1, num_unique_triples(o))}));
}

size_t frag_oz_layout(const Handle* h, int64_t o, int64_t v, int B, char* base, FragOz* W) {
  const int64_t v3 = v * v * v, nt = num_unique_triples(o);
  Carve c{base};
  W->ovvvC = c.d(o * v3);
  W->t2C = c.d(o * o * v * v);
  W->t2C2 = c.d(o * o * v * v);
  W->ooovC = c.d(o * o * o * v);
  W->ovs = c.d(o * v * o * v);
  W->stride = (3 * v3 + 3) / 4 * 4;
  W->G = reinterpret_cast<float2*>(c.d(B * W->stride));
  W->SG = reinterpret_cast<float2*>(c.d(B * W->stride));
  W->epart = c.d((int64_t)B * adjoint_grid(h->num_sms));
  W->shares = c.d(std::max<int64_t>(1, nt));
  for (int k = 0; k < 3; ++k) W->slices[k] = c.take(tc_slices_bytes((int)o, (int)v) + 1024);
  return c.off + 1024;
}

struct ProjArgs {
  AdjArgs a;              // inputs
  SliceExps x0, xa, xb;   // scales of the input slices, of (ovvvC, t2C, ., ooovC) and of t2C2's t2L
  const float2 *G, *SG;   // pairs relative to the largest scale of their products
  int64_t stride;
  double* epart;          // [slot][gridDim.x]
  double* shares;
  int64_t t0;
  int n;
  Triple t[FRAG_MAX_BATCH];
};

// the projected block's scale: the largest of its eight products'
__device__ __forceinline__ int sg_exp(const ProjArgs& A, int p, int q, int r) {
  const int o = A.a.o, rq = r * o + q, rp = r * o + p, nqr = q * o + r, npr = p * o + r;
  int e = max(A.xa.e_ovvv[p] + A.x0.e_t2[rq], A.x0.e_ovvv[p] + A.xa.e_t2[rq]);
  e = max(e, max(A.xa.e_ovvv[q] + A.x0.e_t2[rp], A.x0.e_ovvv[q] + A.xa.e_t2[rp]));
  e = max(e, max(A.xb.e_t2L[p] + A.x0.e_nooT[nqr], A.x0.e_t2L[p] + A.xa.e_nooT[nqr]));
  return max(e, max(A.xb.e_t2L[q] + A.x0.e_nooT[npr], A.x0.e_t2L[q] + A.xa.e_nooT[npr]));
}

// A block at the six positions of an orbit, as float64: the pairs are exact in it.
// The conversions are integer operations (pair_double): as float64 ones they would
// be 36 of 120 per orbit.
__device__ __forceinline__ void orbit_block(const float2* __restrict__ G, const int64_t* at, int e, double* g) {
  float2 x[6];
  bool other = false;
#pragma unroll
  for (int n = 0; n < 6; ++n) x[n] = __ldg(G + at[n]);
#pragma unroll
  for (int n = 0; n < 6; ++n) g[n] = pair_double(x[n].x, x[n].y, e, &other);
  if (other) {
    const double scale = ldexp(1.0, e);
#pragma unroll
    for (int n = 0; n < 6; ++n) g[n] = pair_convert(x[n].x, x[n].y, scale);
  }
}
// W~ (or S W~): G_0 at a position, G_1 at its cyclic successor, G_2 at the one after
__device__ __forceinline__ void orbit_w(const float2* G, int64_t v3, const int* e, const int64_t* at, double* W) {
  constexpr int r1[6] = {3, 5, 1, 4, 0, 2}, r2[6] = {4, 2, 5, 0, 3, 1};
  double g[6];
  orbit_block(G, at, e[0], W);
  orbit_block(G + v3, at, e[1], g);
#pragma unroll
  for (int n = 0; n < 6; ++n) W[n] += g[r1[n]];
  orbit_block(G + 2 * v3, at, e[2], g);
#pragma unroll
  for (int n = 0; n < 6; ++n) W[n] += g[r2[n]];
}

// per-block sums of (S W~) R[V] / D over the orbits of each slot, in float64 from
// the pairs on.  Its two lanes per SM and cycle bound it, some 70 operations per
// orbit, 30 of the 47 ms it takes at nocc=16 nvir=120 (160 ms in all; with W~, D and
// the sums in FP32 pairs 30 and 143, at 48 bits; one thread per element of v^3, a
// sixth of them an orbit, 102 of 320).  Four blocks per SM: 47 ms, two 52.
__global__ void __launch_bounds__(256, 4) k_proj_batch(const __grid_constant__ ProjArgs A) {
  __shared__ double red[8];
  const int slot = blockIdx.y;
  const Triple T = A.t[slot];
  const AdjArgs& a = A.a;
  const int eg[3] = {g_exp(A.x0, a.o, T.i, T.j, T.k), g_exp(A.x0, a.o, T.j, T.k, T.i), g_exp(A.x0, a.o, T.k, T.i, T.j)};
  const int es[3] = {sg_exp(A, T.i, T.j, T.k), sg_exp(A, T.j, T.k, T.i), sg_exp(A, T.k, T.i, T.j)};
  const float2 *G = A.G + slot * A.stride, *SG = A.SG + slot * A.stride;
  const int64_t v = a.v, v3 = v * v * v, steps = orbit_steps(a.v);
  const OrbitTile tile = orbit_tile();
  const int64_t ox = (int64_t)a.o * v;  // doubles between the rows of ovs
  const double *ovs_ij = a.ovs + T.i * v * ox + T.j * v, *ovs_jk = a.ovs + T.j * v * ox + T.k * v,
               *ovs_ik = a.ovs + T.i * v * ox + T.k * v;
  const double *t1i = a.t1 + T.i * v, *t1j = a.t1 + T.j * v, *t1k = a.t1 + T.k * v;
  const double eo = a.eps_o[T.i] + a.eps_o[T.j] + a.eps_o[T.k];
  double sum = 0.0;
  for (int64_t t = blockIdx.x; t < steps; t += gridDim.x) {
    int x, y, z;
    if (!orbit_at(tile, t, a.v, &x, &y, &z)) continue;
    double V[6], S[6], RV[6];
    int64_t at[6];
    orbit_index(v, x, y, z, at);
    orbit_w(G, v3, eg, at, V);
    const int p[6][3] = {{x, y, z}, {x, z, y}, {y, x, z}, {y, z, x}, {z, x, y}, {z, y, x}};
#pragma unroll
    for (int n = 0; n < 6; ++n) {  // V = W~ + Y
      const int q0 = p[n][0], q1 = p[n][1], q2 = p[n][2];
      V[n] = fma(ovs_ij[(int64_t)q0 * ox + q1], t1k[q2], V[n]);
      V[n] = fma(ovs_jk[(int64_t)q1 * ox + q2], t1i[q0], V[n]);
      V[n] = fma(ovs_ik[(int64_t)q0 * ox + q2], t1j[q1], V[n]);
    }
    r_orbit_sums(V, RV);
    orbit_w(SG, v3, es, at, S);
    const unsigned distinct = orbit_distinct(x, y, z);
    double e = 0.0;
#pragma unroll
    for (int n = 0; n < 6; ++n)
      if (distinct >> n & 1u) e = fma(S[n], RV[n], e);
    const double D = eo - a.eps_v[x] - a.eps_v[y] - a.eps_v[z];
    sum = fma(e, recip_newton(D, recip_newton(D, recip_seed(D))), sum);
  }
  for (int off = 16; off > 0; off >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += red[w];
    A.epart[(int64_t)slot * gridDim.x + blockIdx.x] = t;
  }
}

// the slots' shares: (m / 3) (1 / 3) times their block sums in a fixed order
__global__ void __launch_bounds__(256) k_proj_shares(const __grid_constant__ ProjArgs A, int nblk) {
  __shared__ double red[8];
  const int slot = blockIdx.x;
  double s = 0.0;
  for (int e = threadIdx.x; e < nblk; e += 256) s += A.epart[(int64_t)slot * nblk + e];
  for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += red[w];
    A.shares[A.t0 + slot] = t * ((double)A.t[slot].m / 9.0);
  }
}

te_status run_frag_oz(Handle* h, const te_cluster* c, const double* cf, const FragOz& W, int B, cudaStream_t s) {
  const int o = (int)c->nocc, v = (int)c->nvir;
  const int64_t v2 = (int64_t)v * v, v3 = v2 * v, nt = num_unique_triples(o);
  cudaError_t e = transform_inputs(h, c, cf, W.ovvvC, W.t2C, W.t2C2, W.ooovC, s);
  if (e != cudaSuccess) return fail(TE_ECUDA, "transform launch: %s", cudaGetErrorString(e));
  // exact-slice planes: the inputs; (ovvvC, t2C, ooovC) for ovvv, t2 and nooT;
  // t2C2 for t2L
  SliceSet S0{}, SA{}, SB{};
  te_cluster ca = *c, cb = *c;
  ca.ovvv = W.ovvvC;
  ca.t2 = W.t2C;
  ca.ooov = W.ooovC;
  cb.t2 = W.t2C2;
  te_status st = tc_prepare_slices(c, W.slices[0], &S0, h->num_sms, s, 4, h->d_err, 0, &h->n_launches);
  if (st == TE_OK) st = tc_prepare_slices(&ca, W.slices[1], &SA, h->num_sms, s, 4, nullptr, 0, &h->n_launches);
  if (st == TE_OK) st = tc_prepare_slices(&cb, W.slices[2], &SB, h->num_sms, s, 4, nullptr, 0, &h->n_launches);
  if (st != TE_OK) return st;
  Prepared P{};
  P.ovs = W.ovs;
  e = launch_prep_fp64(c, &P, s);
  ++h->n_launches;
  if (e != cudaSuccess) return fail(TE_ECUDA, "prep: %s", cudaGetErrorString(e));
  // the six segment views of each slice set, encoded once
  VtBank bank;
  bank.n = 0;
  int m0[6], mA[6], mB[6];
  const int NT = vt_ntile(v, true);
  if ((st = vt_slice_maps(&bank, S0, o, v, NT, m0)) != TE_OK) return st;
  if ((st = vt_slice_maps(&bank, SA, o, v, NT, mA)) != TE_OK) return st;
  if ((st = vt_slice_maps(&bank, SB, o, v, NT, mB)) != TE_OK) return st;
  const int grid = adjoint_grid(h->num_sms);
  ProjArgs A{};
  A.a.o = o;
  A.a.v = v;
  A.a.ovs = W.ovs;
  A.a.t1 = c->t1;
  A.a.eps_o = c->eps_o;
  A.a.eps_v = c->eps_v;
  A.x0 = SliceExps{S0.e_ovvv, S0.e_t2, S0.e_t2L, S0.e_nooT};
  A.xa = SliceExps{SA.e_ovvv, SA.e_t2, SA.e_t2L, SA.e_nooT};
  A.xb = SliceExps{SB.e_ovvv, SB.e_t2, SB.e_t2L, SB.e_nooT};
  A.G = W.G;
  A.SG = W.SG;
  A.stride = W.stride;
  A.epart = W.epart;
  A.shares = W.shares;
  std::vector<Triple> trip = unique_triples(o);
  VtBuild* bp = new (std::nothrow) VtBuild;
  if (!bp) return fail(TE_ENOMEM, "view GEMM tables");
  VtBuild& b = *bp;
  struct Del {
    VtBuild* b;
    ~Del() { delete b; }
  } del{bp};
  for (int64_t t0 = 0; t0 < nt; t0 += B) {
    A.n = (int)std::min<int64_t>(B, nt - t0);
    A.t0 = t0;
    // per G block (p, q, r): the block itself (S1..S4 of the input slices) and
    // its projection SG (two products per segment, one operand transformed)
    vt_begin(&b, S0.ns, true);
    for (int x = 0; x < A.n; ++x) {
      const Triple T = A.t[x] = trip[t0 + x];
      for (int gi = 0; gi < 3; ++gi) {
        int pp, qq, rr;
        if (gi == 0) { pp = T.i; qq = T.j; rr = T.k; }
        else if (gi == 1) { pp = T.j; qq = T.k; rr = T.i; }
        else { pp = T.k; qq = T.i; rr = T.j; }
        const int f_p[3] = {0, 0, pp}, f_q[3] = {0, 0, qq};
        const int t_qr[3] = {0, qq, rr}, t_pr[3] = {0, pp, rr}, n_rq[3] = {0, rr, qq}, n_rp[3] = {0, rr, pp};
        const int64_t rq = (int64_t)rr * o + qq, rp = (int64_t)rr * o + pp;
        const int64_t nqr = (int64_t)qq * o + rr, npr = (int64_t)pp * o + rr;
        auto seg = [&](int ma, int mb, int K, const int* fa, const int* fb, const int* ea, const int* eb) {
          vt_seg(&b, vt_use(&b, bank, ma), vt_use(&b, bank, mb), 1, K, fa, fb, ea, eb, 1);
        };
        vt_job(&b, v, v, v, 8, 16, NT, W.G + x * W.stride + gi * v3, v2, v, 1, VT_PAIR);
        seg(m0[0], m0[4], v, f_p, t_qr, S0.e_ovvv + pp, S0.e_t2 + rq);
        seg(m0[1], m0[4], v, f_q, t_pr, S0.e_ovvv + qq, S0.e_t2 + rp);
        seg(m0[3], m0[5], o, f_p, n_rq, S0.e_t2L + pp, S0.e_nooT + nqr);
        seg(m0[2], m0[5], o, f_q, n_rp, S0.e_t2L + qq, S0.e_nooT + npr);
        vt_job(&b, v, v, v, 8, 16, NT, W.SG + x * W.stride + gi * v3, v2, v, 1, VT_PAIR);
        seg(mA[0], m0[4], v, f_p, t_qr, SA.e_ovvv + pp, S0.e_t2 + rq);   // ovvvC[p] t2[r,q]
        seg(m0[0], mA[4], v, f_p, t_qr, S0.e_ovvv + pp, SA.e_t2 + rq);   // ovvv[p] t2C[r,q]
        seg(mA[1], m0[4], v, f_q, t_pr, SA.e_ovvv + qq, S0.e_t2 + rp);   // ovvvC[q] t2[r,p]
        seg(m0[1], mA[4], v, f_q, t_pr, S0.e_ovvv + qq, SA.e_t2 + rp);   // ovvv[q] t2C[r,p]
        seg(mB[3], m0[5], o, f_p, n_rq, SB.e_t2L + pp, S0.e_nooT + nqr);  // t2LC[p] nooT[q][r]
        seg(m0[3], mA[5], o, f_p, n_rq, S0.e_t2L + pp, SA.e_nooT + nqr);  // t2L[p] nooTC[q][r]
        seg(mB[2], m0[5], o, f_q, n_rp, SB.e_t2L + qq, S0.e_nooT + npr);  // t2LC[q] nooT[p][r]
        seg(m0[2], mA[5], o, f_q, n_rp, S0.e_t2L + qq, SA.e_nooT + npr);  // t2L[q] nooTC[p][r]
      }
    }
    if ((st = vt_finish(&b, h->num_sms, nullptr, 0, nullptr)) != TE_OK) return st;
    if ((st = vt_launch(h, &b, s)) != TE_OK) return st;
    k_proj_batch<<<dim3((unsigned)grid, (unsigned)A.n), 256, 0, s>>>(A);
    k_proj_shares<<<(unsigned)A.n, 256, 0, s>>>(A, grid);
    h->n_launches += 2;
    e = cudaGetLastError();
    if (e != cudaSuccess) return fail(TE_ECUDA, "projected energy launch: %s", cudaGetErrorString(e));
  }
  return TE_OK;
}

}  // namespace

// The usual batch, then triple by triple where memory is short.
std::vector<size_t> frag_bytes(const Handle* h, int64_t o, int64_t v, te_precision p) {
  if (p == TE_FP64) {
    FragWork W;
    return {frag_layout(o, v, nullptr, &W)};
  }
  FragOz W;
  return {frag_oz_layout(h, o, v, frag_batch(o, v), nullptr, &W), frag_oz_layout(h, o, v, 1, nullptr, &W)};
}

te_status run_frag(Handle* h, const te_cluster* c, const double* cf, te_precision p, double* e_out,
                   double* e_triples, cudaStream_t s) {
  const int o = (int)c->nocc, v = (int)c->nvir;
  const int64_t nt = num_unique_triples(o);
  size_t form = 0;
  te_status st = acquire_workspace(h, frag_bytes(h, o, v, p), &form);
  if (st != TE_OK) return st;
  FragOz Z;
  const int B = form == 0 ? frag_batch(o, v) : 1;
  st = ensure_triples_public(h, o);
  if (st != TE_OK) return st;
  char* base = reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(h->ws) + 1023) & ~uintptr_t(1023));
  const double* shares;
  if (p == TE_FP64) {
    FragWork W;
    frag_layout(o, v, base, &W);
    shares = W.shares;
    st = run_frag_fp64(h, c, cf, W, s);
  } else {
    frag_oz_layout(h, o, v, B, base, &Z);
    shares = Z.shares;
    st = run_frag_oz(h, c, cf, Z, B, s);
  }
  if (st != TE_OK) return st;
  cudaError_t e = cudaSuccess;
  if (e_triples && nt > 0)
    e = cudaMemcpyAsync(e_triples, shares, sizeof(double) * nt, cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess && e_out) {
    if (nt > 0) {
      e = launch_reduce_total(shares, nt, e_out, s);
      ++h->n_launches;
    } else {
      e = cudaMemsetAsync(e_out, 0, sizeof(double), s);
    }
  }
  if (e != cudaSuccess) return fail(TE_ECUDA, "projected energy launch: %s", cudaGetErrorString(e));
  return TE_OK;
}

}  // namespace te
