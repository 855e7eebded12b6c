// Float64 path: operand preparation and the W~ contractions on the DFMA units.
//
// The connected triples of one occupied triple (i,j,k) (Eq. W times D,
// supplement section on (T)) are assembled from three "G" blocks,
//
//   W~_{ijk}[a,b,c] = G(i,j,k)[a,b,c] + G(j,k,i)[b,c,a] + G(k,i,j)[c,a,b],
//
//   G(p,q,r)[x,y,z] = sum_d ( (px|yd) t_{rq}^{zd} + (qy|xd) t_{rp}^{zd} )
//                   - sum_l ( t_{lp}^{yx} (ql|rz) + t_{lq}^{xy} (pl|rz) )
//
// written as one GEMM per (p,q,r): rows (x,y) flattened (v^2), columns z (v),
// and a K axis made of four segments:
//   S1  A = ovvv[p, x, y, :]        B = t2[r, q, z, :]            K = v
//   S2  A = ovvv[q, y, x, :]        B = t2[r, p, z, :]            K = v
//   S3  A = t2L[p, y, x, :]         B = nooT[q, r, z, :]          K = o
//   S4  A = t2L[q, x, y, :]         B = nooT[p, r, z, :]          K = o
// with t2L[q][x][y][l] = t2[l,q,x,y] and nooT[p][r][z][l] = -ooov[p,l,r,z].
// Each of the six terms of the permutation operator P appears exactly once in
// the three G blocks (S1/S2 carry the sum over d, S3/S4 the sum over l).
#include <algorithm>

#include "dfma_tile.cuh"
#include "te_internal.h"

namespace te {

// ---------------------------------------------------------------------------
// preparation kernels (float64)
// ---------------------------------------------------------------------------

__global__ void k_prep_t2L(const double* __restrict__ t2, double* __restrict__ t2L, int o, int v) {
  const int64_t n = (int64_t)o * v * v * o;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int l = (int)(idx % o);
    int64_t rest = idx / o;
    const int b = (int)(rest % v);
    rest /= v;
    const int a = (int)(rest % v);
    const int q = (int)(rest / v);
    t2L[idx] = t2[(((int64_t)l * o + q) * v + a) * v + b];
  }
}

__global__ void k_prep_nooT(const double* __restrict__ ooov, double* __restrict__ nooT, int o, int v) {
  const int64_t n = (int64_t)o * o * v * o;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int l = (int)(idx % o);
    int64_t rest = idx / o;
    const int z = (int)(rest % v);
    rest /= v;
    const int r = (int)(rest % o);
    const int p = (int)(rest / o);
    nooT[idx] = -ooov[(((int64_t)p * o + l) * o + r) * v + z];
  }
}

__global__ void k_prep_ovs(const double* __restrict__ ovov, double* __restrict__ ovs, int o, int v) {
  const int64_t n = (int64_t)o * v * o * v;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int b = (int)(idx % v);
    int64_t rest = idx / v;
    const int j = (int)(rest % o);
    rest /= o;
    const int a = (int)(rest % v);
    const int i = (int)(rest / v);
    ovs[idx] = 0.5 * (ovov[idx] + ovov[(((int64_t)j * v + b) * o + i) * v + a]);
  }
}

static int grid_for(int64_t n) {
  int64_t g = (n + 255) / 256;
  if (g > 8192) g = 8192;
  if (g < 1) g = 1;
  return (int)g;
}

cudaError_t launch_prep_fp64(const te_cluster* c, Prepared* P, cudaStream_t s) {
  const int o = (int)c->nocc, v = (int)c->nvir;
  // the tensor-core adjoint reads its own slice planes: no float64 t2L / nooT copies
  if (P->t2L) k_prep_t2L<<<grid_for((int64_t)o * v * v * o), 256, 0, s>>>(c->t2, P->t2L, o, v);
  if (P->nooT) k_prep_nooT<<<grid_for((int64_t)o * o * v * o), 256, 0, s>>>(c->ooov, P->nooT, o, v);
  k_prep_ovs<<<grid_for((int64_t)o * v * o * v), 256, 0, s>>>(c->ovov, P->ovs, o, v);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// DFMA GEMM: one CTA = 32 RM rows (x,y) x 8 NB columns z of one G block
// (dfma_tile.cuh).  The float64 units bound it: 12 v^3 (v + o) flops per triple
// at 1.25 TFLOP/s (3.3 ms).  nocc=8 nvir=40, whole energy: 8.18 ms with 64 x 64 tiles
// (40 columns on 64, K of 40 and 8 on 48 and 16), 3.85 ms with the picked one.
// ---------------------------------------------------------------------------

template <int RM, int NB>
__global__ void __launch_bounds__(DT_THREADS)
k_gemm_fp64(const double* __restrict__ ovvv, const double* __restrict__ t2,
            const double* __restrict__ t2L, const double* __restrict__ nooT,
            const Triple* __restrict__ triples, int64_t t0, int o, int v,
            double* __restrict__ gbuf) {
  __shared__ DfmaSmem<RM, NB> S;
  constexpr int TM = 32 * RM, TN = 8 * NB;
  const int tid = threadIdx.x;
  const int slot = blockIdx.z / 3;
  const int g = blockIdx.z % 3;
  const Triple T = triples[t0 + slot];
  int p, q, r;
  if (g == 0) { p = T.i; q = T.j; r = T.k; }
  else if (g == 1) { p = T.j; q = T.k; r = T.i; }
  else { p = T.k; q = T.i; r = T.j; }
  const int64_t v2 = (int64_t)v * v;
  const int64_t v3 = v2 * v;
  const int64_t row0 = (int64_t)blockIdx.x * TM;
  const int col0 = blockIdx.y * TN;

  // loader: 16 threads per row take its 16 k; the row's (x, y) stays the same
  const int lk = tid & 15, lr = tid >> 4;
  int rx[2 * RM], ry[2 * RM];
#pragma unroll
  for (int i = 0; i < 2 * RM; ++i) {
    const int64_t R = row0 + lr + 16 * i;
    rx[i] = R < v2 ? (int)(R / v) : -1;
    ry[i] = R < v2 ? (int)(R % v) : 0;
  }
  double acc[RM][NB];
#pragma unroll
  for (int a = 0; a < RM; ++a)
#pragma unroll
    for (int b = 0; b < NB; ++b) acc[a][b] = 0.0;

  for (int seg = 0; seg < 4; ++seg) {
    const bool swap = seg == 1 || seg == 2;  // rows (y, x)
    const double *A, *B;
    int K;
    if (seg == 0) { A = ovvv + (int64_t)p * v3; B = t2 + ((int64_t)r * o + q) * v2; K = v; }
    else if (seg == 1) { A = ovvv + (int64_t)q * v3; B = t2 + ((int64_t)r * o + p) * v2; K = v; }
    else if (seg == 2) { A = t2L + (int64_t)p * v2 * o; B = nooT + ((int64_t)q * o + r) * v * o; K = o; }
    else { A = t2L + (int64_t)q * v2 * o; B = nooT + ((int64_t)p * o + r) * v * o; K = o; }
    for (int k0 = 0; k0 < K; k0 += DT_K) {
      const int kk = k0 + lk;
#pragma unroll
      for (int i = 0; i < 2 * RM; ++i) {
        const int64_t row = swap ? (int64_t)ry[i] * v + rx[i] : (int64_t)rx[i] * v + ry[i];
        S.a[lk][lr + 16 * i] = (rx[i] >= 0 && kk < K) ? A[row * K + kk] : 0.0;
      }
#pragma unroll
      for (int i = 0; i < (TN + 15) / 16; ++i) {
        const int c = lr + 16 * i;
        if (c < TN) S.b[lk][c] = (col0 + c < v && kk < K) ? B[(int64_t)(col0 + c) * K + kk] : 0.0;
      }
      __syncthreads();
      dfma_chunk<RM, NB>(S, min(DT_K, K - k0), acc);
      __syncthreads();
    }
  }
  double* out = gbuf + ((int64_t)slot * 3 + g) * v3;
  const int tx = tid & 7, ty = tid >> 3;
#pragma unroll
  for (int a = 0; a < RM; ++a) {
    const int64_t Ro = row0 + ty + 32 * a;
    if (Ro >= v2) continue;
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const int z = col0 + tx + 8 * b;
      if (z < v) out[Ro * v + z] = acc[a][b];
    }
  }
}

// (K = 2 (v + o): only its length against the staging matters to the pick)
static DfmaPick gemm_fp64_pick(int64_t v, int nslots, int num_sms) {
  return dfma_pick(v * v, v, 2 * v + 16, 3LL * nslots, std::max(1, num_sms), 0, false);
}

cudaError_t launch_gemm_fp64(const Prepared* P, const Triple* d_triples, int64_t t0, int nslots,
                             double* gbuf, int num_sms, cudaStream_t s) {
  const DfmaPick t = gemm_fp64_pick(P->v, nslots, num_sms);
  const dim3 grid((unsigned)t.tiles_m, (unsigned)t.tiles_n, (unsigned)(3 * nslots));
  dfma_dispatch(t, [&](auto rm, auto nb) {
    k_gemm_fp64<decltype(rm)::value, decltype(nb)::value>
        <<<grid, DT_THREADS, 0, s>>>(P->ovvv, P->t2, P->t2L, P->nooT, d_triples, t0, P->o, P->v, gbuf);
  });
  return cudaGetLastError();
}

}  // namespace te
