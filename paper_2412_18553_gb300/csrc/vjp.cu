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
#include <atomic>
#include <cuda_bf16.h>

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
// (ia|jb), 29.1 ms now.
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

// Split count for a GEMM of `tiles` output tiles and K steps: about two
// blocks per SM, each split at least 8 K steps; the scratch holds `cap`
// doubles.
static int num_splits(int64_t tiles, int64_t K, int64_t MN, int num_sms, int64_t cap) {
  const int64_t steps = (K + DT_K - 1) / DT_K;
  int64_t want = (2LL * num_sms + tiles - 1) / tiles;
  want = std::min<int64_t>(want, std::max<int64_t>(1, steps / 8));
  want = std::min<int64_t>(want, std::max<int64_t>(1, cap / std::max<int64_t>(1, MN)));
  return (int)std::max<int64_t>(1, want);
}

cudaError_t gemm_strided(const GemmView& g, int num_sms, double* scratch, int64_t scratch_cap, cudaStream_t s,
                         int64_t* launches) {
  const int64_t M = g.M1 * g.M2, K = g.K1 * g.K2;
  const DfmaPick t = dfma_pick(M, g.N);
  const int ns = num_splits(t.tiles_m * t.tiles_n, K, M * g.N, num_sms, scratch_cap);
  const int64_t steps = (K + DT_K - 1) / DT_K;
  const int kchunk = (int)(((steps + ns - 1) / ns) * DT_K);
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
// exact-slice strided GEMM on the tensor cores (mma.sync, BF16 -> FP32):
//   C[m,n] (+)= alpha 2^(ea + eb) sum_k A[m,k] B[k,n]
// A and B are NS BF16 slice planes each (slice s at base + s * plane; NS = 4,
// or 5 for 35-bit operands), read through the same two-index strided views as
// the float64 kernel.  The slice products a_i b_j with i + j <= NS - 1 (ten,
// or fifteen) go to three FP32 accumulators:
// level 0 and level 1 exactly (K <= 1024 per block keeps their partial sums
// integer multiples of the level's unit below 2^24), the higher levels
// approximately; each block's sums go to float64 once, at its end.
// ---------------------------------------------------------------------------


constexpr int OZ_BM = 64, OZ_BN = 64, OZ_BK = 32, OZ_KMAX = 1024;
constexpr int OZ_THREADS = 256;  // eight warps, each 32 x 16 outputs
constexpr int OZ_LD = OZ_BK + 8;  // padded row (bf16): conflict-free fragment loads

__device__ __forceinline__ void mma_bf16_16816(float* d, const uint32_t* a, const uint32_t* b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// Tiles of 64 x 64 outputs, 32 k per stage, two stages in flight (cp.async).
// Each operand tile sits in shared memory k-major ([row][k]) when its view is
// contiguous along k, else row-major ([k][row]) when contiguous along its rows
// (columns); 16-byte chunks of eight BF16 values are copied asynchronously
// where the view allows, element by element otherwise.
template <bool AK, bool BK, int NS>
struct OzTile {
  static constexpr int A = AK ? OZ_BM * OZ_LD : OZ_BK * (OZ_BM + 8);
  static constexpr int B = BK ? OZ_BN * OZ_LD : OZ_BK * (OZ_BN + 8);
  static constexpr int STAGE = NS * (A + B);  // elements
  static constexpr size_t BYTES = 2 * STAGE * sizeof(__nv_bfloat16);
};

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// four 8 x 8 BF16 matrices from shared memory, as stored / transposed
__device__ __forceinline__ void ldsm_x4(uint32_t* r, const __nv_bfloat16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((uint32_t)__cvta_generic_to_shared(p)));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t* r, const __nv_bfloat16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((uint32_t)__cvta_generic_to_shared(p)));
}

// Eight elements (rows r + e step_r, k + e step_k) of every slice, element by
// element, zero outside the view: ragged edges and views without a
// contiguous index.  Rolled loops, so the pipelined loop stays small enough
// for the instruction cache.
__device__ __forceinline__ void oz_fill_slow(const __nv_bfloat16* __restrict__ src, int64_t ps, __nv_bfloat16* dst,
                                          int dps, int ns, int r, int k, int step_r, int step_k, int R, int ke,
                                          int R2, int64_t r1s, int64_t r2s, int K2, int64_t k1s, int64_t k2s) {
#pragma unroll 1
  for (int e = 0; e < 8; ++e) {
    const int rr = r + e * step_r, kk = k + e * step_k;
    const bool ok = rr < R && kk < ke;
    const int64_t off =
        ok ? (int64_t)(rr / R2) * r1s + (int64_t)(rr % R2) * r2s + (int64_t)(kk / K2) * k1s + (int64_t)(kk % K2) * k2s
           : 0;
#pragma unroll 1
    for (int sl = 0; sl < ns; ++sl) dst[sl * dps + e] = ok ? src[off + sl * ps] : __float2bfloat16_rn(0.f);
  }
}

template <bool AK, bool BK, int NS>
__global__ void __launch_bounds__(OZ_THREADS, 2) k_gemm_oz2(OzView g, int kchunk, double* __restrict__ part,
                                                            int a_vec, int b_vec) {
  using T = OzTile<AK, BK, NS>;
  extern __shared__ __align__(16) unsigned char oz_smem[];
  __nv_bfloat16* smem = reinterpret_cast<__nv_bfloat16*>(oz_smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int M = (int)(g.M1 * g.M2), N = (int)g.N, K2 = (int)g.K2;
  const int m0 = blockIdx.x * OZ_BM, n0 = blockIdx.y * OZ_BN;
  const int kb = blockIdx.z * kchunk, ke = min((int)(g.K1 * g.K2), kb + kchunk);
  const int nst = (ke - kb + OZ_BK - 1) / OZ_BK;

  auto a_row = [&](int m) { return (int64_t)(m / (int)g.M2) * g.a_m1 + (int64_t)(m % (int)g.M2) * g.a_m2; };
  auto a_kof = [&](int k) { return (int64_t)(k / K2) * g.a_k1 + (int64_t)(k % K2) * g.a_k2; };
  auto b_kof = [&](int k) { return (int64_t)(k / K2) * g.b_k1 + (int64_t)(k % K2) * g.b_k2; };
  // 256 chunks of 8 elements per slice and operand, OZ_CH per thread; the row
  // (column) part of a chunk's offset is the same at every stage
  constexpr int OZ_CH = 256 / OZ_THREADS;
  int64_t a_roff[OZ_CH];
#pragma unroll
  for (int c2 = 0; c2 < OZ_CH; ++c2) {
    const int c = tid + OZ_THREADS * c2;
    const int m = AK ? m0 + (c >> 2) : m0 + (c & 7) * 8;
    a_roff[c2] = m < M ? a_row(m) : 0;
  }

  // one 8-element chunk: elements e = 0..7 along the tile's contiguous direction
  auto load_stage = [&](int buf, int k0) {
    __nv_bfloat16* As = smem + buf * T::STAGE;
    __nv_bfloat16* Bs = As + NS * T::A;
#pragma unroll
    for (int c2 = 0; c2 < OZ_CH; ++c2) {
      const int c = tid + OZ_THREADS * c2;
      // ---- A ----
      {
        int m, k, step_m, step_k;  // first element and the step between the 8
        __nv_bfloat16* dst0;
        if (AK) {
          m = m0 + (c >> 2);
          k = k0 + (c & 3) * 8;
          step_m = 0;
          step_k = 1;
          dst0 = As + (c >> 2) * OZ_LD + (c & 3) * 8;
        } else {
          k = k0 + (c >> 3);
          m = m0 + (c & 7) * 8;
          step_m = 1;
          step_k = 0;
          dst0 = As + (c >> 3) * (OZ_BM + 8) + (c & 7) * 8;
        }
        const bool full = a_vec && (AK ? (m < M && k + 8 <= ke) : (k < ke && m + 8 <= M));
        if (full) {
          const __nv_bfloat16* src = g.A + a_roff[c2] + a_kof(k);
#pragma unroll
          for (int sl = 0; sl < NS; ++sl) cp_async16(dst0 + sl * T::A, src + sl * g.a_ps);
        } else {
          oz_fill_slow(g.A, g.a_ps, dst0, T::A, NS, m, k, step_m, step_k, M, ke, (int)g.M2, g.a_m1, g.a_m2, K2,
                       g.a_k1, g.a_k2);
        }
      }
      // ---- B ----
      {
        int n, k, step_n, step_k;
        __nv_bfloat16* dst0;
        if (BK) {
          n = n0 + (c >> 2);
          k = k0 + (c & 3) * 8;
          step_n = 0;
          step_k = 1;
          dst0 = Bs + (c >> 2) * OZ_LD + (c & 3) * 8;
        } else {
          k = k0 + (c >> 3);
          n = n0 + (c & 7) * 8;
          step_n = 1;
          step_k = 0;
          dst0 = Bs + (c >> 3) * (OZ_BN + 8) + (c & 7) * 8;
        }
        const bool full = b_vec && (BK ? (n < N && k + 8 <= ke) : (k < ke && n + 8 <= N));
        if (full) {
          const __nv_bfloat16* src = g.B + (int64_t)n * g.b_n + b_kof(k);
#pragma unroll
          for (int sl = 0; sl < NS; ++sl) cp_async16(dst0 + sl * T::B, src + sl * g.b_ps);
        } else {
          oz_fill_slow(g.B, g.b_ps, dst0, T::B, NS, n, k, step_n, step_k, N, ke, 1, g.b_n, 0, K2, g.b_k1, g.b_k2);
        }
      }
    }
  };

  const int wm = (warp & 1) * 32, wn = (warp >> 1) * 16;
  const int gq = lane >> 2, tq = lane & 3;
  float acc[3][2][2][4];
#pragma unroll
  for (int l = 0; l < 3; ++l)
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[l][i][j][q] = 0.f;

  if (nst > 0) load_stage(0, kb);
  cp_async_commit();
  for (int st = 0; st < nst; ++st) {
    if (st + 1 < nst) load_stage((st + 1) & 1, kb + (st + 1) * OZ_BK);
    cp_async_commit();
    cp_async_wait1();  // every group but the newest: this stage's copies have landed
    __syncthreads();
    const __nv_bfloat16* As = smem + (st & 1) * T::STAGE;
    const __nv_bfloat16* Bs = As + NS * T::A;
#pragma unroll
    for (int kk = 0; kk < OZ_BK; kk += 16) {
      // ldmatrix: lane l addresses row (l & 7) of 8 x 8 matrix (l >> 3)
      const int lr = lane & 7, lm = lane >> 3;
      uint32_t bf[NS][2][2];
#pragma unroll
      for (int sl = 0; sl < NS; ++sl) {
        // matrices: (cols 0-7, k kk), (cols 0-7, k kk+8), (cols 8-15, k kk), (cols 8-15, k kk+8)
        const __nv_bfloat16* b = Bs + sl * T::B;
        uint32_t t[4];
        const int cb = wn + (lm >> 1) * 8;
        if (BK) ldsm_x4(t, b + (cb + lr) * OZ_LD + kk + (lm & 1) * 8);
        else ldsm_x4_t(t, b + (kk + lr + (lm & 1) * 8) * (OZ_BN + 8) + cb);
        bf[sl][0][0] = t[0];
        bf[sl][0][1] = t[1];
        bf[sl][1][0] = t[2];
        bf[sl][1][1] = t[3];
      }
#pragma unroll
      for (int sa = 0; sa < NS; ++sa) {
        uint32_t af[2][4];  // A slice sa, loaded when its products are due
        const __nv_bfloat16* a = As + sa * T::A;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int r = wm + i * 16;
          // matrices: (rows r, k kk), (rows r+8, k kk), (rows r, k kk+8), (rows r+8, k kk+8)
          if (AK) ldsm_x4(af[i], a + (r + lr + (lm & 1) * 8) * OZ_LD + kk + (lm >> 1) * 8);
          else ldsm_x4_t(af[i], a + (kk + lr + (lm >> 1) * 8) * (OZ_BM + 8) + r + (lm & 1) * 8);
        }
#pragma unroll
        for (int sb = 0; sb < NS - sa; ++sb) {
          const int lev = sa + sb == 0 ? 0 : (sa + sb == 1 ? 1 : 2);
#pragma unroll
          for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j) mma_bf16_16816(acc[lev][i][j], af[i], bf[sb][j]);
        }
      }
    }
    __syncthreads();  // the buffer is refilled two stages on
  }
  const double scale = ldexp(g.alpha, *g.ea + *g.eb);
  // this thread's four output rows (i, half h) and their offsets in C
  int64_t crow[2][2];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
      const int m = m0 + wm + i * 16 + gq + hh * 8;
      crow[i][hh] = m < M ? (int64_t)(m / (int)g.M2) * g.c_m1 + (int64_t)(m % (int)g.M2) * g.c_m2 : 0;
    }
  // Per 16-row half: every old value of C is loaded before any store, so the
  // loads overlap (a store could otherwise alias the next load).
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    double val[2][4], old[2][4];
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int m = m0 + wm + i * 16 + gq + (q >> 1) * 8;
        const int n = n0 + wn + j * 8 + 2 * tq + (q & 1);
        val[j][q] = scale * (((double)acc[0][i][j][q] + (double)acc[1][i][j][q]) + (double)acc[2][i][j][q]);
        old[j][q] = (!part && !g.overwrite && m < M && n < N) ? g.C[crow[i][q >> 1] + n * g.c_n] : 0.0;
      }
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int m = m0 + wm + i * 16 + gq + (q >> 1) * 8;
        const int n = n0 + wn + j * 8 + 2 * tq + (q & 1);
        if (m >= M || n >= N) continue;
        if (part) part[((int64_t)blockIdx.z * M + m) * N + n] = val[j][q];
        else g.C[crow[i][q >> 1] + n * g.c_n] = old[j][q] + val[j][q];
      }
  }
}

// C[m,n] += sum_z part[z][m][n], z in order (alpha is already applied)
__global__ void k_splitk_add_oz(OzView g, int nsplit, const double* __restrict__ part) {
  const int M = (int)(g.M1 * g.M2);
  const int64_t MN = (int64_t)M * g.N;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < MN; e += (int64_t)gridDim.x * blockDim.x) {
    double s = 0.0;  // in split order; unrolled so that many loads are in flight
#pragma unroll 16
    for (int z = 0; z < nsplit; ++z) s += part[z * MN + e];
    const int m = (int)(e / g.N), n = (int)(e % g.N);
    double* cp = g.C + (int64_t)(m / (int)g.M2) * g.c_m1 + (int64_t)(m % (int)g.M2) * g.c_m2 + n * g.c_n;
    *cp = g.overwrite ? s : *cp + s;
  }
}

template <bool AK, bool BK, int NS>
static cudaError_t launch_oz2(const OzView& g, dim3 grid, int kchunk, double* part, int av, int bv, cudaStream_t s) {
  const size_t bytes = OzTile<AK, BK, NS>::BYTES;
  static std::atomic<unsigned long long> opted{0};  // devices this instantiation may use `bytes` on
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = 1ull << (dev & 63);
  if (!(opted.load() & bit)) {
    e = cudaFuncSetAttribute(k_gemm_oz2<AK, BK, NS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return e;
    opted.fetch_or(bit);
  }
  k_gemm_oz2<AK, BK, NS><<<grid, OZ_THREADS, bytes, s>>>(g, kchunk, part, av, bv);
  return cudaGetLastError();
}

// K in splits of at most OZ_KMAX (exactness), more when the output has few
// tiles: the K chunk per split (a multiple of OZ_BK)
static int oz_kchunk(int64_t M, int64_t N, int64_t K, int num_sms) {
  const int64_t tm = (M + OZ_BM - 1) / OZ_BM, tn = (N + OZ_BN - 1) / OZ_BN;
  const int64_t steps = (K + OZ_BK - 1) / OZ_BK;
  int64_t ns = std::max<int64_t>((K + OZ_KMAX - 1) / OZ_KMAX, (2LL * num_sms + tm * tn - 1) / (tm * tn));
  ns = std::min<int64_t>(ns, std::max<int64_t>(1, steps / 4));
  ns = std::max<int64_t>(ns, (K + OZ_KMAX - 1) / OZ_KMAX);
  return (int)(((steps + ns - 1) / ns) * OZ_BK);
}

int64_t gemm_oz_scratch(int64_t M, int64_t N, int64_t K, int num_sms) {
  const int kchunk = oz_kchunk(M, N, K, num_sms);
  const int64_t nsplit = (K + kchunk - 1) / kchunk;
  return nsplit > 1 ? nsplit * M * N : 0;
}

cudaError_t gemm_oz(const OzView& g, int num_sms, double* scratch, int64_t scratch_cap, cudaStream_t s,
                           int64_t* launches) {
  const int64_t M = g.M1 * g.M2, K = g.K1 * g.K2;
  const int64_t tm = (M + OZ_BM - 1) / OZ_BM, tn = (g.N + OZ_BN - 1) / OZ_BN;
  const int kchunk = oz_kchunk(M, g.N, K, num_sms);
  const int nsplit = (int)((K + kchunk - 1) / kchunk);
  if (nsplit > 1 && (int64_t)nsplit * M * g.N > scratch_cap) return cudaErrorInvalidValue;
  dim3 grid((unsigned)tm, (unsigned)tn, (unsigned)nsplit);
  // tile orientation per operand: k-major if the view is contiguous along k,
  // else row-major if contiguous along its rows (columns), else k-major
  // element by element
  auto al16 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  const bool a_k = g.a_ps % 8 == 0 && al16(g.A) &&
                   ((g.K2 == 1 && g.a_k1 == 1) || (g.K2 % 8 == 0 && g.a_k2 == 1 && g.a_k1 % 8 == 0)) &&
                   (g.a_m1 % 8 == 0 || g.M1 == 1) && (g.a_m2 % 8 == 0 || g.M2 == 1);
  const bool a_m = !a_k && g.a_ps % 8 == 0 && al16(g.A) &&
                   ((g.M2 == 1 && g.a_m1 == 1) || (g.M2 % 8 == 0 && g.a_m2 == 1 && g.a_m1 % 8 == 0)) &&
                   g.a_k1 % 8 == 0 && (g.K2 == 1 || g.a_k2 % 8 == 0);
  const bool b_k = g.b_ps % 8 == 0 && al16(g.B) &&
                   ((g.K2 == 1 && g.b_k1 == 1) || (g.K2 % 8 == 0 && g.b_k2 == 1 && g.b_k1 % 8 == 0)) && g.b_n % 8 == 0;
  const bool b_n = !b_k && g.b_ps % 8 == 0 && al16(g.B) && g.b_n == 1 && g.b_k1 % 8 == 0 &&
                   (g.K2 == 1 || g.b_k2 % 8 == 0);
  double* pp = nsplit > 1 ? scratch : nullptr;
  const bool AK = !a_m, BK = !b_n;
  const int av = (a_k || a_m) ? 1 : 0, bv = (b_k || b_n) ? 1 : 0;
  cudaError_t err;
  if (g.ns == 5) {
    if (AK && BK) err = launch_oz2<true, true, 5>(g, grid, kchunk, pp, av, bv, s);
    else if (AK) err = launch_oz2<true, false, 5>(g, grid, kchunk, pp, av, bv, s);
    else if (BK) err = launch_oz2<false, true, 5>(g, grid, kchunk, pp, av, bv, s);
    else err = launch_oz2<false, false, 5>(g, grid, kchunk, pp, av, bv, s);
  } else if (g.ns == 0 || g.ns == 4) {
    if (AK && BK) err = launch_oz2<true, true, 4>(g, grid, kchunk, pp, av, bv, s);
    else if (AK) err = launch_oz2<true, false, 4>(g, grid, kchunk, pp, av, bv, s);
    else if (BK) err = launch_oz2<false, true, 4>(g, grid, kchunk, pp, av, bv, s);
    else err = launch_oz2<false, false, 4>(g, grid, kchunk, pp, av, bv, s);
  } else {
    return cudaErrorInvalidValue;
  }
  if (err != cudaSuccess) return err;
  ++*launches;
  if (nsplit > 1) {
    const int64_t MN = M * g.N;
    k_splitk_add_oz<<<(unsigned)std::min<int64_t>((MN + 255) / 256, 4096), 256, 0, s>>>(g, nsplit, scratch);
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
    e = launch_gemm_fp64(&P, h->d_triples, t, 1, W.G, s);
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
