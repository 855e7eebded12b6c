// Adjoint of E(T): dE/d(eps_o, eps_v, ovvv, ooov, ovov, t1, t2), in float64
// (DFMA contractions; the exact-slice adjoint is in adjoint_tc.cu).
//
// E = sum over unique occupied triples t of (m_t/3) e_t,
//   e_t = sum_{abc} W~[abc] R[V][abc] / D[abc],  V = W~ + Y,
// with R acting on the virtual indices at fixed ijk (equal to R on the
// occupied ones at fixed abc).  R's coefficient pattern (4, 3-cycles +1,
// transpositions -2) is symmetric and D is invariant under permutations of
// abc, so with w_t = gE m_t / 3:
//   dW~ = w_t R[2 W~ + Y] / D,   dY = w_t R[W~] / D,   dD = -w_t W~ R[V] / D^2.
// W~[a,b,c] = G0[a,b,c] + G1[b,c,a] + G2[c,a,b] gives dG0[x,y,z] = dW~[x,y,z],
// dG1[x,y,z] = dW~[z,x,y], dG2[x,y,z] = dW~[y,z,x]; each G block
//   G(p,q,r)[x,y,z] = sum_d ovvv[p,x,y,d] t2[r,q,z,d] + sum_d ovvv[q,y,x,d] t2[r,p,z,d]
//                   - sum_l t2[l,p,y,x] ooov[q,l,r,z] - sum_l t2[l,q,x,y] ooov[p,l,r,z]
// back-propagates through eight GEMMs (two per K segment).  Y = ovs(ia,jb) t1(kc)
// + ovs(jb,kc) t1(ia) + ovs(ia,kc) t1(jb) with ovs = (ovov + ovov^T)/2 gives the
// ovov and t1 parts.  Triples are processed one after another on the stream
// and every accumulation has a fixed order, so the gradient is deterministic.
#include <algorithm>
#include <initializer_list>
#include <vector>

#include "adjoint_tc.cuh"
#include "dfma_tile.cuh"
#include "strided.h"
#include "te_internal.h"

namespace te {

// ---------------------------------------------------------------------------
// per-triple adjoint of the energy epilogue, one thread per ordered (a,b,c)
// ---------------------------------------------------------------------------

// blocks of the adjoint epilogue: a fixed number per device, so the orbits
// each block takes, and every partial sum, do not depend on the cluster
int adjoint_grid(int num_sms) { return std::min(4 * std::max(1, num_sms), 8192); }

// Threads stride over the orbits a >= b >= c (v(v+1)(v+2)/6 of them): W~ and Y
// are formed once per orbit and every distinct element of the orbit gets its
// dW~, dY and dD.  1/D is Newton's iteration x <- x (2 - D x) from an FP32
// seed, twice (relative error below 2^-90 before rounding): float64 division
// costs several times more on GB300's float64 units.  Each block writes its
// energy and dD partial sums to epart, dpart[blockIdx.x].
__global__ void __launch_bounds__(256) k_adjoint(AdjArgs A) {
  __shared__ double red[8], redd[8];
  const int64_t v = A.v;
  const int64_t norb = v * (v + 1) * (v + 2) / 6;
  const double eo = A.eps_o[A.i] + A.eps_o[A.j] + A.eps_o[A.k];
  double contrib = 0.0, dsum = 0.0;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < norb; t += (int64_t)gridDim.x * blockDim.x) {
    int a, b, c;
    orbit_abc(t, &a, &b, &c);
    double W[6], Y[6], RW[6], RY[6];
    int64_t idx[6];
    orbit_values(A, a, b, c, W, Y);
    orbit_index(v, a, b, c, idx);
    r_orbit(W, RW);
    r_orbit(Y, RY);
    const unsigned distinct = orbit_distinct(a, b, c);
    const double D = eo - A.eps_v[a] - A.eps_v[b] - A.eps_v[c];
    double rD = (double)__frcp_rn((float)D);
    rD = fma(rD, fma(-D, rD, 1.0), rD);
    rD = fma(rD, fma(-D, rD, 1.0), rD);
    const double q = A.w * rD;
#pragma unroll
    for (int n = 0; n < 6; ++n) {
      if (!(distinct >> n & 1u)) continue;
      const double RV = RW[n] + RY[n];
      const double dw = q * (2.0 * RW[n] + RY[n]);
      const double dd = -q * W[n] * RV * rD;
      A.dW[idx[n]] = dw;
      A.dY[idx[n]] = q * RW[n];
      A.dD[idx[n]] = dd;
      dsum += dd;
      contrib += W[n] * RV * rD;
    }
  }
  for (int off = 16; off > 0; off >>= 1) {
    contrib += __shfl_down_sync(0xffffffffu, contrib, off);
    dsum += __shfl_down_sync(0xffffffffu, dsum, off);
  }
  if ((threadIdx.x & 31) == 0) {
    red[threadIdx.x >> 5] = contrib;
    redd[threadIdx.x >> 5] = dsum;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0, sd = 0.0;
    for (int w = 0; w < 8; ++w) {
      s += red[w];
      sd += redd[w];
    }
    A.epart[blockIdx.x] = s;
    A.dpart[blockIdx.x] = sd;
  }
}

// ---------------------------------------------------------------------------
// generic strided float64 GEMM:  C[m,n] += alpha sum_k A[m,k] B[k,n]
// m = (m1, m2), k = (k1, k2), each index with its own stride.  Outputs with
// few tiles (the contractions over a virtual pair, K = v^2) split K over
// blockIdx.z into fixed ranges; the partial tiles go to a scratch array and
// are added in split order by k_splitk_add, so the result is deterministic.
// ---------------------------------------------------------------------------


// One CTA = 32 RM x 8 NB outputs of one K range (dfma_tile.cuh).  a_fast,
// b_fast: the loader's threads run along k when the view is contiguous there,
// else along the rows (columns).  With `sym` (the output is symmetric, both
// operands the same view, no K split) only the tiles that reach m >= n are
// computed, and each of their elements with m >= n is written at (m, n) and at
// (n, m): a product of the same two factors in the same K order, so the
// mirrored bits are those the other half would have had.  The float64 units
// bound every launch; eight clusters' MP2 step (nocc 8 .. 20, nvir = 8 nocc,
// three contractions each): 56.1 ms with 64 x 64 tiles and both halves of
// (ia|jb), 26 ms now.
template <int RM, int NB>
__global__ void __launch_bounds__(DT_THREADS) k_gemm_strided(const __grid_constant__ GemmView g, int kchunk,
                                                             double* __restrict__ part, int a_fast, int b_fast,
                                                             int sym) {
  constexpr int TM = 32 * RM, TN = 8 * NB;
  const int m0 = blockIdx.x * TM, n0 = blockIdx.y * TN;
  if (sym && m0 + TM <= n0) return;
  __shared__ DfmaSmem<RM, NB> S;
  const int tid = threadIdx.x;
  const int M = (int)(g.M1 * g.M2), N = (int)g.N, K = (int)(g.K1 * g.K2), K2 = (int)g.K2, M2 = (int)g.M2;
  const int kb = blockIdx.z * kchunk, ke = min(K, kb + kchunk);
  double acc[RM][NB];
#pragma unroll
  for (int a = 0; a < RM; ++a)
#pragma unroll
    for (int b = 0; b < NB; ++b) acc[a][b] = 0.0;
  for (int k0 = kb; k0 < ke; k0 += DT_K) {
#pragma unroll
    for (int i = 0; i < 2 * RM; ++i) {
      const int e = tid + DT_THREADS * i;
      const int kk = a_fast ? e & 15 : e / TM, r = a_fast ? e >> 4 : e % TM;
      const int m = m0 + r, k = k0 + kk;
      double x = 0.0;
      if (m < M && k < ke) {
        const int m1 = m / M2, k1 = k / K2;
        x = g.A[m1 * g.a_m1 + (m - m1 * M2) * g.a_m2 + k1 * g.a_k1 + (k - k1 * K2) * g.a_k2];
      }
      S.a[kk][r] = x;
    }
#pragma unroll
    for (int i = 0; i < (TN * DT_K + DT_THREADS - 1) / DT_THREADS; ++i) {
      const int e = tid + DT_THREADS * i;
      if (e >= TN * DT_K) break;
      const int kk = b_fast ? e & 15 : e / TN, c = b_fast ? e >> 4 : e % TN;
      const int n = n0 + c, k = k0 + kk;
      double x = 0.0;
      if (n < N && k < ke) {
        const int k1 = k / K2;
        x = g.B[n * g.b_n + k1 * g.b_k1 + (k - k1 * K2) * g.b_k2];
      }
      S.b[kk][c] = x;
    }
    __syncthreads();
    dfma_chunk<RM, NB>(S, min(DT_K, ke - k0), acc);
    __syncthreads();
  }
  const int tx = tid & 7, ty = tid >> 3;
#pragma unroll
  for (int a = 0; a < RM; ++a) {
    const int m = m0 + ty + 32 * a;
    if (m >= M) continue;
    const int64_t crow = (int64_t)(m / M2) * g.c_m1 + (int64_t)(m % M2) * g.c_m2;
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const int n = n0 + tx + 8 * b;
      if (n >= N) continue;
      if (part) {  // split K: this split's tile, row-major [M][N]
        part[((int64_t)blockIdx.z * M + m) * N + n] = acc[a][b];
      } else if (!sym) {
        g.C[crow + n * g.c_n] += g.alpha * acc[a][b];
      } else if (m >= n) {
        const double x = g.alpha * acc[a][b];
        g.C[crow + n * g.c_n] += x;
        if (m > n) g.C[(int64_t)(n / M2) * g.c_m1 + (int64_t)(n % M2) * g.c_m2 + m * g.c_n] += x;
      }
    }
  }
}

// C[m,n] += alpha sum_z part[z][m][n], z in order
__global__ void k_splitk_add(GemmView g, int nsplit, const double* __restrict__ part) {
  const int M = (int)(g.M1 * g.M2);
  const int64_t MN = (int64_t)M * g.N;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < MN; e += (int64_t)gridDim.x * blockDim.x) {
    double s = 0.0;  // in split order; unrolled so that many loads are in flight
#pragma unroll 16
    for (int z = 0; z < nsplit; ++z) s += part[z * MN + e];
    const int m = (int)(e / g.N), n = (int)(e % g.N);
    const int64_t crow = (int64_t)(m / (int)g.M2) * g.c_m1 + (int64_t)(m % (int)g.M2) * g.c_m2;
    g.C[crow + n * g.c_n] += g.alpha * s;
  }
}

cudaError_t gemm_strided(const GemmView& g, int num_sms, double* scratch, int64_t scratch_cap, cudaStream_t s,
                         int64_t* launches) {
  const int64_t M = g.M1 * g.M2, K = g.K1 * g.K2;
  const DfmaPick t = dfma_pick(M, g.N, K, 1, std::max(1, num_sms), scratch_cap, g.symmetric);
  const int64_t steps = (K + DT_K - 1) / DT_K;
  const int kchunk = (int)(((steps + t.nsplit - 1) / t.nsplit) * DT_K);
  const int nsplit = (int)((K + kchunk - 1) / kchunk);
  const dim3 grid((unsigned)t.tiles_m, (unsigned)t.tiles_n, (unsigned)nsplit);
  const bool a_fast = (g.K2 > 1 ? g.a_k2 : g.a_k1) == 1, b_fast = (g.K2 > 1 ? g.b_k2 : g.b_k1) == 1;
  const int sym = g.symmetric && nsplit == 1 ? 1 : 0;
  double* part = nsplit > 1 ? scratch : nullptr;
  dfma_dispatch(t, [&](auto rm, auto nb) {
    k_gemm_strided<decltype(rm)::value, decltype(nb)::value>
        <<<grid, DT_THREADS, 0, s>>>(g, kchunk, part, a_fast ? 1 : 0, b_fast ? 1 : 0, sym);
  });
  ++*launches;
  if (nsplit > 1) {
    const int64_t MN = M * g.N;
    k_splitk_add<<<(unsigned)std::min<int64_t>((MN + 255) / 256, 4096), 256, 0, s>>>(g, nsplit, scratch);
    ++*launches;
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Y and denominator reductions for one triple
// ---------------------------------------------------------------------------

// dOVS[P1][x][P2][y] += sum_z dY[perm(x,y,z)] t1[P3][z]   (one of the three Y terms)
// mode 0: ovs(i,a,j,b) t1(k,c): out (a,b), sum over c; t1 row k
// mode 1: ovs(j,b,k,c) t1(i,a): out (b,c), sum over a; t1 row i
// mode 2: ovs(i,a,k,c) t1(j,b): out (a,c), sum over b; t1 row j
__global__ void k_dovs(int mode, int o, int v, int i, int j, int k, const double* __restrict__ dY,
                       const double* __restrict__ t1, double* __restrict__ dOVS) {
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= (int64_t)v * v) return;
  const int x = (int)(idx / v), y = (int)(idx % v);
  const int64_t V = v;
  double s = 0.0;
  int P1, P2, P3;
  if (mode == 0) {
    P1 = i; P2 = j; P3 = k;
    for (int c = 0; c < v; ++c) s += dY[(x * V + y) * V + c] * t1[(int64_t)P3 * v + c];
  } else if (mode == 1) {
    P1 = j; P2 = k; P3 = i;
    for (int a = 0; a < v; ++a) s += dY[(a * V + x) * V + y] * t1[(int64_t)P3 * v + a];
  } else {
    P1 = i; P2 = k; P3 = j;
    for (int b = 0; b < v; ++b) s += dY[(x * V + b) * V + y] * t1[(int64_t)P3 * v + b];
  }
  dOVS[(((int64_t)P1 * v + x) * o + P2) * v + y] += s;
}

// fixed-order block sum of 256 threads' values; the result is valid in thread 0
__device__ __forceinline__ double block_sum256(double s, double* red) {
  for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < 8; ++w) t += red[w];
  return t;
}

// dt1[P3][z] += sum over the other two indices of dY * ovs (one of the three
// Y terms); one block per z
__global__ void __launch_bounds__(256) k_dt1(int mode, int o, int v, int i, int j, int k,
                                              const double* __restrict__ dY, const double* __restrict__ ovs,
                                              double* __restrict__ dt1) {
  __shared__ double red[8];
  const int z = blockIdx.x;
  const int64_t V = v, n = V * V;
  auto OV = [&](int P1, int a, int P2, int b) { return ovs[(((int64_t)P1 * v + a) * o + P2) * v + b]; };
  double s = 0.0;
  for (int64_t e = threadIdx.x; e < n; e += blockDim.x) {
    const int p = (int)(e / v), q = (int)(e % v);
    if (mode == 0) s += dY[(p * V + q) * V + z] * OV(i, p, j, q);       // t1(k,c): dY[a,b,c] ovs(i,a,j,b)
    else if (mode == 1) s += dY[(z * V + p) * V + q] * OV(j, p, k, q);  // t1(i,a): dY[a,b,c] ovs(j,b,k,c)
    else s += dY[(p * V + z) * V + q] * OV(i, p, k, q);                 // t1(j,b): dY[a,b,c] ovs(i,a,k,c)
  }
  const double t = block_sum256(s, red);
  if (threadIdx.x == 0) {
    const int row = mode == 0 ? k : (mode == 1 ? i : j);
    dt1[(int64_t)row * v + z] += t;
  }
}

// deps_v[x] -= sum_bc dD[x,b,c] + sum_ac dD[a,x,c] + sum_ab dD[a,b,x]; one block per x
__global__ void __launch_bounds__(256) k_deps_v(int v, const double* __restrict__ dD, double* __restrict__ deps_v) {
  __shared__ double red[8];
  const int x = blockIdx.x;
  const int64_t V = v, n = V * V;
  double s = 0.0;
  for (int64_t e = threadIdx.x; e < n; e += blockDim.x) {
    const int p = (int)(e / v), q = (int)(e % v);
    s += dD[(x * V + p) * V + q] + dD[(p * V + x) * V + q] + dD[(p * V + q) * V + x];
  }
  const double t = block_sum256(s, red);
  if (threadIdx.x == 0) deps_v[x] -= t;
}

// deps_o[i], [j], [k] += sum_abc dD, from the adjoint kernel's per-block sums
// (fixed-order block sum)
__global__ void __launch_bounds__(256) k_deps_o(int64_t n, const double* __restrict__ dpart, int i, int j, int k,
                                                 double* __restrict__ deps_o) {
  __shared__ double red[8];
  double s = 0.0;
  for (int64_t e = threadIdx.x; e < n; e += blockDim.x) s += dpart[e];
  for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += red[w];
    deps_o[i] += t;
    deps_o[j] += t;
    deps_o[k] += t;
  }
}

// dovov[P1,x,P2,y] = (dOVS[P1,x,P2,y] + dOVS[P2,y,P1,x]) / 2
__global__ void k_dovov(int o, int v, const double* __restrict__ dOVS, double* __restrict__ dovov) {
  const int64_t n = (int64_t)o * v * o * v;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int y = (int)(idx % v);
    int64_t rest = idx / v;
    const int P2 = (int)(rest % o);
    rest /= o;
    const int x = (int)(rest % v);
    const int P1 = (int)(rest / v);
    dovov[idx] = 0.5 * (dOVS[idx] + dOVS[(((int64_t)P2 * v + y) * o + P1) * v + x]);
  }
}

cudaError_t launch_dovov(int o, int v, const double* dOVS, double* dovov, cudaStream_t s) {
  k_dovov<<<1024, 256, 0, s>>>(o, v, dOVS, dovov);
  return cudaGetLastError();
}

// sum of the adjoint kernel's per-block partials -> one per-triple share
__global__ void __launch_bounds__(256) k_sum_share(const double* __restrict__ part, int64_t n, double scale,
                                                    double* __restrict__ out) {
  __shared__ double red[8];
  double s = 0.0;
  for (int64_t e = threadIdx.x; e < n; e += blockDim.x) s += part[e];
  for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += red[w];
    *out = t * scale;
  }
}

cudaError_t launch_sum_share(const double* part, int64_t n, double scale, double* out, cudaStream_t s) {
  k_sum_share<<<1, 256, 0, s>>>(part, n, scale, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// driver
// ---------------------------------------------------------------------------

struct VjpWork {
  double *t2L, *nooT, *ovs, *G, *dW, *dY, *dD, *dOVS, *epart, *dpart, *shares, *splitk;
};

// doubles of split-K scratch: room for the partial tiles of a v x v output
int64_t splitk_cap(int64_t o, int64_t v) { return 80 * std::max(v * v, o * v); }

size_t vjp_fp64_bytes(int64_t o, int64_t v) {
  const int64_t v3 = v * v * v, nt = num_unique_triples(o);
  const int64_t nblk = std::max<int64_t>((v3 + 255) / 256, 8192);  // at least adjoint_grid's largest
  auto a = [](int64_t n) { return ((size_t)n * 8 + 255) & ~size_t(255); };
  return a(o * v * v * o) + a(o * o * v * o) + a(o * v * o * v) + a(3 * v3) + 3 * a(v3) + a(o * v * o * v) +
         2 * a(nblk) + a(std::max<int64_t>(1, nt)) + a(splitk_cap(o, v)) + 1024;
}

te_status ensure_workspace_public(Handle* h, size_t bytes);
te_status ensure_triples_public(Handle* h, int nocc);

te_status run_vjp_fp64(Handle* h, const te_cluster* c, int64_t t_begin, int64_t t_end, double gE,
                       double* e_out, te_cluster_grad* g, cudaStream_t s) {
  const int o = (int)c->nocc, v = (int)c->nvir;
  const int64_t v2 = (int64_t)v * v, v3 = v2 * v, nt = num_unique_triples(o);
  te_status st = ensure_workspace_public(h, vjp_fp64_bytes(o, v));
  if (st != TE_OK) return st;
  st = ensure_triples_public(h, o);
  if (st != TE_OK) return st;
  char* p = reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(h->ws) + 255) & ~uintptr_t(255));
  auto take = [&](int64_t n) {
    double* r = reinterpret_cast<double*>(p);
    p += ((size_t)n * 8 + 255) & ~size_t(255);
    return r;
  };
  VjpWork W;
  W.t2L = take((int64_t)o * v * v * o);
  W.nooT = take((int64_t)o * o * v * o);
  W.ovs = take((int64_t)o * v * o * v);
  W.G = take(3 * v3);
  W.dW = take(v3);
  W.dY = take(v3);
  W.dD = take(v3);
  W.dOVS = take((int64_t)o * v * o * v);
  const int64_t nblk = std::max<int64_t>((v3 + 255) / 256, adjoint_grid(h->num_sms));
  const int64_t agrid = adjoint_grid(h->num_sms);
  W.epart = take(nblk);
  W.dpart = take(nblk);
  W.shares = take(std::max<int64_t>(1, nt));
  W.splitk = take(splitk_cap(o, v));

  // gradient outputs start at zero
  auto zero = [&](double* ptr, int64_t n) {
    return ptr ? cudaMemsetAsync(ptr, 0, sizeof(double) * n, s) : cudaSuccess;
  };
  cudaError_t e = cudaSuccess;
  e = e ? e : zero(g->eps_o, o);
  e = e ? e : zero(g->eps_v, v);
  e = e ? e : zero(g->ovvv, (int64_t)o * v3);
  e = e ? e : zero(g->ooov, (int64_t)o * o * o * v);
  e = e ? e : zero(g->ovov, (int64_t)o * v * o * v);
  e = e ? e : zero(g->t1, (int64_t)o * v);
  e = e ? e : zero(g->t2, (int64_t)o * o * v2);
  e = e ? e : zero(W.dOVS, (int64_t)o * v * o * v);
  if (e != cudaSuccess) return fail(TE_ECUDA, "memset: %s", cudaGetErrorString(e));

  Prepared P{};
  P.o = o;
  P.v = v;
  P.eps_o = c->eps_o;
  P.eps_v = c->eps_v;
  P.ovvv = c->ovvv;
  P.t2 = c->t2;
  P.t1 = c->t1;
  P.t2L = W.t2L;
  P.nooT = W.nooT;
  P.ovs = W.ovs;
  e = launch_prep_fp64(c, &P, s);
  if (e != cudaSuccess) return fail(TE_ECUDA, "prep: %s", cudaGetErrorString(e));

  std::vector<Triple> trip = unique_triples(o);
  for (int64_t t = t_begin; t < t_end && e == cudaSuccess; ++t) {
    const Triple T = trip[t];
    e = launch_gemm_fp64(&P, h->d_triples, t, 1, W.G, h->num_sms, s);
    if (e != cudaSuccess) break;
    AdjArgs A{};
    A.o = o; A.v = v; A.i = T.i; A.j = T.j; A.k = T.k;
    A.w = gE * (double)T.m / 3.0;
    A.G = W.G; A.ovs = W.ovs; A.t1 = c->t1; A.eps_o = c->eps_o; A.eps_v = c->eps_v;
    A.dW = W.dW; A.dY = W.dY; A.dD = W.dD; A.epart = W.epart; A.dpart = W.dpart;
    k_adjoint<<<(unsigned)agrid, 256, 0, s>>>(A);
    k_sum_share<<<1, 256, 0, s>>>(W.epart, agrid, (double)T.m / 3.0, W.shares + t);
    h->n_launches += 3;
    // back-propagation through the three G blocks; Gamma_g is a strided view of dW~
    for (int gi = 0; gi < 3 && e == cudaSuccess; ++gi) {
      int pp, qq, rr;
      if (gi == 0) { pp = T.i; qq = T.j; rr = T.k; }
      else if (gi == 1) { pp = T.j; qq = T.k; rr = T.i; }
      else { pp = T.k; qq = T.i; rr = T.j; }
      // Gamma[x,y,z] strides (gx, gy, gz)
      int64_t gx, gy, gz;
      if (gi == 0) { gx = v2; gy = v; gz = 1; }        // dW~[x,y,z]
      else if (gi == 1) { gx = v; gy = 1; gz = v2; }   // dW~[z,x,y]
      else { gx = 1; gy = v2; gz = v; }                // dW~[y,z,x]
      const double* t2rq = c->t2 + ((int64_t)rr * o + qq) * v2;
      const double* t2rp = c->t2 + ((int64_t)rr * o + pp) * v2;
      auto run = [&](GemmView gv) {
        if (e == cudaSuccess) e = gemm_strided(gv, h->num_sms, W.splitk, splitk_cap(o, v), s, &h->n_launches);
      };
      if (g->ovvv) {
        // (a) dovvv[p,x,y,d] += sum_z G[x,y,z] t2[r,q,z,d]
        run(GemmView{W.dW, t2rq, g->ovvv + (int64_t)pp * v3, v, v, v, v, 1, gx, gy, gz, 0, v, 0, 1, v2, v, 1, 1.0});
        // (b) dovvv[q,y,x,d] += sum_z G[x,y,z] t2[r,p,z,d]
        run(GemmView{W.dW, t2rp, g->ovvv + (int64_t)qq * v3, v, v, v, v, 1, gx, gy, gz, 0, v, 0, 1, v, v2, 1, 1.0});
      }
      if (g->t2) {
        // (c) dt2[r,q,z,d] += sum_xy G[x,y,z] ovvv[p,x,y,d]
        run(GemmView{W.dW, c->ovvv + (int64_t)pp * v3, g->t2 + ((int64_t)rr * o + qq) * v2, v, 1, v, v, v, gz, 0,
                     gx, gy, v2, v, 1, v, 0, 1, 1.0});
        // (d) dt2[r,p,z,d] += sum_xy G[x,y,z] ovvv[q,y,x,d]
        run(GemmView{W.dW, c->ovvv + (int64_t)qq * v3, g->t2 + ((int64_t)rr * o + pp) * v2, v, 1, v, v, v, gz, 0,
                     gx, gy, v, v2, 1, v, 0, 1, 1.0});
        // (e) dt2[l,p,y,x] -= sum_z G[x,y,z] ooov[q,l,r,z]
        run(GemmView{W.dW, c->ooov + ((int64_t)qq * o * o + rr) * v, g->t2 + (int64_t)pp * v2, v, v, o, v, 1, gx,
                     gy, gz, 0, 1, 0, (int64_t)o * v, 1, v, (int64_t)o * v2, -1.0});
        // (g) dt2[l,q,x,y] -= sum_z G[x,y,z] ooov[p,l,r,z]
        run(GemmView{W.dW, c->ooov + ((int64_t)pp * o * o + rr) * v, g->t2 + (int64_t)qq * v2, v, v, o, v, 1, gx,
                     gy, gz, 0, 1, 0, (int64_t)o * v, v, 1, (int64_t)o * v2, -1.0});
      }
      if (g->ooov) {
        // (f) dooov[q,l,r,z] -= sum_xy t2[l,p,y,x] G[x,y,z]
        run(GemmView{c->t2 + (int64_t)pp * v2, W.dW, g->ooov + ((int64_t)qq * o * o + rr) * v, o, 1, v, v, v,
                     (int64_t)o * v2, 0, 1, v, gx, gy, gz, (int64_t)o * v, 0, 1, -1.0});
        // (h) dooov[p,l,r,z] -= sum_xy t2[l,q,x,y] G[x,y,z]
        run(GemmView{c->t2 + (int64_t)qq * v2, W.dW, g->ooov + ((int64_t)pp * o * o + rr) * v, o, 1, v, v, v,
                     (int64_t)o * v2, 0, v, 1, gx, gy, gz, (int64_t)o * v, 0, 1, -1.0});
      }
    }
    if (e != cudaSuccess) break;
    // disconnected term and denominators
    const unsigned gb2 = (unsigned)((v2 + 255) / 256);
    for (int mode = 0; mode < 3; ++mode) {
      if (g->ovov) k_dovs<<<gb2, 256, 0, s>>>(mode, o, v, T.i, T.j, T.k, W.dY, c->t1, W.dOVS);
      if (g->t1) k_dt1<<<(unsigned)v, 256, 0, s>>>(mode, o, v, T.i, T.j, T.k, W.dY, W.ovs, g->t1);
    }
    if (g->eps_v) k_deps_v<<<(unsigned)v, 256, 0, s>>>(v, W.dD, g->eps_v);
    if (g->eps_o) k_deps_o<<<1, 256, 0, s>>>(agrid, W.dpart, T.i, T.j, T.k, g->eps_o);
    h->n_launches += 8;
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && g->ovov) {
    e = launch_dovov(o, v, W.dOVS, g->ovov, s);
    ++h->n_launches;
  }
  if (e == cudaSuccess && e_out) {
    e = launch_reduce_total(W.shares + t_begin, t_end - t_begin, e_out, s);
    ++h->n_launches;
  }
  if (e != cudaSuccess) return fail(TE_ECUDA, "vjp launch: %s", cudaGetErrorString(e));
  return TE_OK;
}

}  // namespace te
