// The MP2 step that precedes (T) in the SIE workflow, for a batch of clusters
// (supplement section on bath-natural-orbital construction):
//
//   (ia|jb)   = sum_P B[P,i,a] B[P,j,b]                       (density fitting)
//   t_ij^ab   = -(ia|jb) / D_ij^ab,  D_ij^ab = e_a + e_b - e_i - e_j
//   gamma_ab  = 2 sum_ij sum_c t_ij^ac (2 t_ij^bc - t_ij^cb)
//   gamma_ij  = 2 delta_ij - 2 sum_k sum_ab t_ik^ab (2 t_jk^ab - t_jk^ba)
//   populations: the eigenvalues of gamma_oo and gamma_vv (BNO populations)
//
// The three contractions are GEMMs over two-index views (strided.h).  The
// (ia|jb) contraction runs in float64 on the DFMA units or, in the exact-slice
// mode, in exact BF16 slices on the tensor cores (Bov scaled by one power of
// two and cut into four 7-bit slices, K in blocks of 128 that keep the
// level-0/1 sums exact).  The density contractions run in float64 in both
// modes: their K spans the amplitudes' whole dynamic range (o^2 v and o v^2
// terms), which one scale per array would resolve only to ~1e-6 of the
// largest entry; they cost o/naux and o/v of the first.  With T~ = 2t - t^(ab
// swapped), both density blocks are single contractions against T~:
//   gamma_vv[a,b] = 2 sum_{(ij),c} t[ij,a,c] T~[ij,b,c]
//   gamma_oo[i,j] = 2 delta_ij - 2 sum_{k,(ab)} t[i,k,ab] T~[j,k,ab]
// The eigenvalues come from a Householder reduction to tridiagonal form (one
// block per matrix, in shared memory up to order 167) and bisection with Sturm
// counts (one thread per eigenvalue), float64 throughout; two launches take the
// matrices of up to 32 clusters, whose density blocks stay in the workspace until
// then.
#include <cuda_bf16.h>

#include <algorithm>
#include <memory>
#include <new>

#include "strided.h"
#include "te_internal.h"
#include "view_tc.h"

namespace te {

te_status ensure_workspace_public(Handle* h, size_t bytes);

namespace {

static int grid_of(int64_t n) { return (int)std::min<int64_t>(std::max<int64_t>(1, (n + 255) / 256), 8192); }

// t[i,j,a,b] = -ovov[i,a,j,b] / D, T~[i,j,a,b] = 2 t[i,j,a,b] - t[i,j,b,a]
// (D is symmetric in a, b, so t[i,j,b,a] = -ovov[i,b,j,a] / D)
__global__ void k_mp2_amplitudes(const double* __restrict__ ovov, const double* __restrict__ eps_o,
                                 const double* __restrict__ eps_v, int o, int v, double* __restrict__ t2,
                                 double* __restrict__ tt) {
  const int64_t n = (int64_t)o * o * v * v;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int b = (int)(idx % v);
    int64_t r = idx / v;
    const int a = (int)(r % v);
    r /= v;
    const int j = (int)(r % o);
    const int i = (int)(r / o);
    const double D = (eps_v[a] + eps_v[b]) - (eps_o[i] + eps_o[j]);
    const double t = -ovov[(((int64_t)i * v + a) * o + j) * v + b] / D;
    const double ts = -ovov[(((int64_t)i * v + b) * o + j) * v + a] / D;
    t2[idx] = t;
    tt[idx] = 2.0 * t - ts;
  }
}

// gamma_oo starts at 2 on the diagonal, 0 elsewhere
__global__ void k_two_identity(double* __restrict__ g, int o) {
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < o * o; idx += gridDim.x * blockDim.x)
    g[idx] = (idx / o == idx % o) ? 2.0 : 0.0;
}

// One symmetric matrix for the eigensolver: the source (n x n), the output
// eigenvalues (n, ascending), n doubles each for the tridiagonal form and a
// global working copy (n x n) for an order too large for shared memory (null
// otherwise).
struct EigJob {
  double* a;
  const double* src;
  double* out;
  double *d, *e;  // diagonal; squares of the off-diagonal; both of the matrix times 2^-e[n - 1]
  int n;
};

// Orders up to this one keep their working copy in shared memory: 167^2
// doubles, two vectors and the partial sums fit the 227 KB of one block.
constexpr int kEigSmemN = 167;
constexpr int EIG_THREADS = 512;

struct EigJobs {
  int count;
  EigJob j[64];
};

// Shared memory of one job: the vectors v and w, the partial sums, then its
// working copy unless it has a global one.
__host__ __device__ inline size_t eig_vec_doubles(int n) { return 2 * (size_t)n + (n > EIG_THREADS ? n : EIG_THREADS); }
__host__ __device__ inline size_t eig_smem_bytes(const EigJob& j) {
  return 8 * (eig_vec_doubles(j.n) + (j.a ? 0 : (size_t)j.n * j.n));
}

__device__ __forceinline__ double warp_sum(double x) {
  for (int d = 16; d > 0; d >>= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
  return x;
}

// Householder reduction of the symmetric part (A + A^T) / 2 (a density computed
// in exact slices is symmetric only to about 1e-9 of its scale), scaled by a
// power of two to entries below 1: step k takes x = A[k+1.., k], v = x + sign(x_0)
// |x| e_0, beta = 1 / (|x|^2 + |x_0| |x|), p = beta A v, w = p - (beta / 2) (v . p)
// v, and A <- A - v w^T - w v^T on the trailing block; the subdiagonal entry is
// -sign(x_0) |x|.
// About n^3 float64 operations on two lanes per cycle of one SM: 1 ms at n = 160.
// (A parallel-order cyclic Jacobi solver, 24 ms for the sixteen matrices of eight
// clusters nocc 8 .. 20, nvir = 8 nocc, was bound by the same two lanes with
// six sweeps of 4 n^3; this and the bisection take 3.0 ms (1.8 and 1.2).)
__global__ void __launch_bounds__(EIG_THREADS, 1) k_tridiag(const __grid_constant__ EigJobs J) {
  const EigJob& jb = J.j[blockIdx.x];
  const int n = jb.n, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  extern __shared__ __align__(16) unsigned char eig_smem[];
  double* v = reinterpret_cast<double*>(eig_smem);
  double* w = v + n;
  double* part = w + n;
  double* A = jb.a ? jb.a : v + eig_vec_doubles(n);
  __shared__ double sh[2];
  __shared__ unsigned int top;
  if (tid == 0) top = 0u;
  __syncthreads();
  unsigned int m = 0;
  for (int64_t e = tid; e < (int64_t)n * n; e += EIG_THREADS) {
    const int r = (int)(e / n), c = (int)(e % n);
    const double x = 0.5 * jb.src[e] + 0.5 * jb.src[(int64_t)c * n + r];
    A[e] = x;
    m = max(m, (unsigned int)__double2hiint(x) & 0x7FFFFFFFu);
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if (lane == 0) atomicMax(&top, m);
  __syncthreads();
  const int ex = top == 0u ? 0 : (int)(top >> 20) - 1022;  // 2^ex > max |a|
  const double sc = ldexp(1.0, -ex);
  for (int64_t e = tid; e < (int64_t)n * n; e += EIG_THREADS) A[e] *= sc;
  __syncthreads();
  for (int k = 0; k + 1 < n; ++k) {
    const int na = n - k - 1;  // order of the trailing block
    const double* row = A + (int64_t)k * n + k + 1;
    if (warp == 0) {
      double s = 0.0;
      for (int i = lane; i < na; i += 32) s = fma(row[i], row[i], s);
      s = warp_sum(s);
      const double x0 = row[0], nx = sqrt(s);
      // a block of one entry is tridiagonal already; so is a column below 1e-100
      const double beta = na > 1 && s > 1e-200 ? 1.0 / (s + fabs(x0) * nx) : 0.0;
      const double alpha = na > 1 ? copysign(nx, -x0) : x0;
      for (int i = lane; i < na; i += 32) v[i] = i == 0 ? x0 - alpha : row[i];
      if (lane == 0) {
        sh[0] = beta;
        jb.d[k] = A[(int64_t)k * n + k];
        jb.e[k] = alpha * alpha;
      }
    }
    __syncthreads();
    const double beta = sh[0];
    if (beta == 0.0) {
      __syncthreads();
      continue;
    }
    double* T = A + (int64_t)(k + 1) * n + k + 1;  // trailing block, row stride n
    // p = A v: rows split into as many parts as there are threads for
    const int parts = na < EIG_THREADS ? EIG_THREADS / na : 1;
    for (int t = tid; t < parts * na; t += EIG_THREADS) {
      const int q = t / na, i = t - q * na, j0 = na * q / parts, j1 = na * (q + 1) / parts;
      double s0 = 0.0, s1 = 0.0;
      int j = j0;
      for (; j + 1 < j1; j += 2) {  // A is symmetric: its rows read along i
        s0 = fma(T[(int64_t)j * n + i], v[j], s0);
        s1 = fma(T[(int64_t)(j + 1) * n + i], v[j + 1], s1);
      }
      if (j < j1) s0 = fma(T[(int64_t)j * n + i], v[j], s0);
      part[t] = s0 + s1;
    }
    __syncthreads();
    if (warp == 0) {
      double s = 0.0;
      for (int i = lane; i < na; i += 32) {
        double p = part[i];
        for (int q = 1; q < parts; ++q) p += part[q * na + i];
        p *= beta;
        w[i] = p;
        s = fma(p, v[i], s);
      }
      s = 0.5 * beta * warp_sum(s);
      for (int i = lane; i < na; i += 32) w[i] = fma(-s, v[i], w[i]);
    }
    __syncthreads();
    for (int i = warp; i < na; i += EIG_THREADS / 32) {
      const double vi = -v[i], wi = -w[i];
      for (int j = lane; j < na; j += 32) T[(int64_t)i * n + j] = fma(vi, w[j], fma(wi, v[j], T[(int64_t)i * n + j]));
    }
    __syncthreads();
  }
  if (tid == 0) {
    jb.d[n - 1] = A[(int64_t)n * n - 1];
    jb.e[n - 1] = (double)ex;
  }
}

// Eigenvalue number m (ascending) of a job's tridiagonal matrix by bisection: a
// thread per eigenvalue, a warp per block (a warp alone on its SM has both
// float64 lanes).  The count of eigenvalues below x is that of the sign changes
// of the leading minors p_i = (d_i - x) p_{i-1} - e_{i-1}^2 p_{i-2} (three float64
// operations a step; the quotients' form takes six with a reciprocal: 2.97
// against 1.20 ms at n = 160).  A minor below 2^-90 of the last one counts as
// -2^-90 of it; pairs are rescaled by a power of two.  All threads start from one interval and
// take the same branch at the same x, so the results ascend.
__global__ void __launch_bounds__(32) k_bisect(const __grid_constant__ EigJobs J) {
  const EigJob& jb = J.j[blockIdx.y];
  const int n = jb.n, lane = threadIdx.x, m = blockIdx.x * 32 + lane;
  if (blockIdx.x * 32 >= n) return;
  extern __shared__ __align__(16) unsigned char eig_smem[];
  double* d = reinterpret_cast<double*>(eig_smem);
  double* e2 = d + n;
  double lo = 1e300, hi = -1e300;
  for (int i = lane; i < n; i += 32) {
    d[i] = jb.d[i];
    e2[i] = i + 1 < n ? jb.e[i] : 0.0;
  }
  __syncwarp();
  for (int i = lane; i < n; i += 32) {  // Gershgorin discs
    const double r = (i > 0 ? sqrt(e2[i - 1]) : 0.0) + sqrt(e2[i]);
    lo = fmin(lo, d[i] - r);
    hi = fmax(hi, d[i] + r);
  }
  for (int k = 16; k > 0; k >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, k));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, k));
  }
  const double pad = 1e-15 * fmax(fabs(lo), fabs(hi)) + 1e-300;
  lo -= pad;
  hi += pad;
  // to 2^-58 of the first interval, the matrix's norm: up to n times its largest
  // entry (all entries equal), 2^-46 of it at the largest order
  for (int it = 0; it < 58; ++it) {
    const double x = 0.5 * (lo + hi);
    int below = 0;
    double p1 = 1.0, p0 = 1.0, e = 0.0;
    for (int i = 0; i < n; ++i) {
      double p = fma(d[i] - x, p1, -(e * p0));
      int h = __double2hiint(p);
      const int h1 = __double2hiint(p1);
      if ((h & 0x7FF00000) + (90 << 20) < (h1 & 0x7FF00000)) {
        h = (int)(((unsigned int)h1 ^ 0x80000000u) - (90u << 20));
        p = __hiloint2double(h, __double2loint(p1));
      }
      below += (h ^ h1) < 0 ? 1 : 0;
      p0 = p1;
      p1 = p;
      const int ex = ((h >> 20) & 0x7FF) - 1023;
      if (ex > 300 || ex < -300) {
        p1 = __hiloint2double(h - ex * (1 << 20), __double2loint(p1));
        p0 = __hiloint2double(h1 - ex * (1 << 20), __double2loint(p0));
      }
      e = e2[i];
    }
    if (below > m) hi = x;
    else lo = x;
  }
  if (m < n) jb.out[m] = ldexp(0.5 * (lo + hi), (int)jb.e[n - 1]);
}

}  // namespace


// Doubles of split-K partial tiles for the float64 contractions, which fit their
// split counts to what they are given.
static int64_t mp2_scratch(int64_t o, int64_t v) {
  return std::max<int64_t>(splitk_cap(o, v), 80LL * std::max(o * o, v * v));
}
static int64_t mp2_pitch(int64_t naux) { return (naux + 7) / 8 * 8; }  // rows of the slices: steps of 16 bytes

static size_t al256(size_t b) { return (b + 255) & ~size_t(255); }

// Bytes of workspace one cluster uses while its contractions run (the largest
// is allocated; the next cluster reuses it).
static size_t mp2_shared_bytes(int64_t o, int64_t v, int64_t naux, bool oz) {
  // split-K partial tiles of the densities; before them, of (ia|jb) or (4 x 2 B per
  // element) the slices of Bov
  return al256((size_t)std::max<int64_t>(mp2_scratch(o, v), oz ? mp2_pitch(naux) * o * v : 0) * 8);
}
static size_t mp2_bytes(int64_t o, int64_t v, int64_t naux, bool oz) {
  const size_t ovov = (size_t)o * v * o * v, t2n = (size_t)o * o * v * v;
  return al256(ovov * 8) + 2 * al256(t2n * 8) + mp2_shared_bytes(o, v, naux, oz) + (oz ? al256(64) : 0);
}

// Bytes one cluster keeps until its group's eigensolver launch: the gamma
// blocks (when the caller did not ask for them) and global working copies for
// orders above kEigSmemN.
static size_t mp2_keep_bytes(int64_t o, int64_t v) {
  size_t b = al256((size_t)o * o * 8) + al256((size_t)v * v * 8);
  if (o > kEigSmemN) b += al256((size_t)o * o * 8);
  if (v > kEigSmemN) b += al256((size_t)v * v * 8);
  return b;
}


// The tridiagonal forms of one cluster.  A group's live where its contractions had
// their transient arrays: the eigensolver runs after the last of them.
static size_t mp2_tri_bytes(int64_t o, int64_t v) { return al256((size_t)o * 16) + al256((size_t)v * 16); }

// Clusters per eigensolver launch: two matrices each, 64 jobs.
constexpr int64_t kMp2Group = 32;

static cudaError_t launch_eig(EigJobs* jobs, cudaStream_t s) {
  size_t bytes = 16;
  int nmax = 1;
  for (int k = 0; k < jobs->count; ++k) {
    bytes = std::max(bytes, eig_smem_bytes(jobs->j[k]));
    nmax = std::max(nmax, jobs->j[k].n);
  }
  cudaError_t e = cudaFuncSetAttribute(k_tridiag, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  k_tridiag<<<jobs->count, EIG_THREADS, bytes, s>>>(*jobs);
  const size_t b2 = (size_t)nmax * 16;
  e = cudaFuncSetAttribute(k_bisect, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)b2);
  if (e != cudaSuccess) return e;
  k_bisect<<<dim3((unsigned)((nmax + 31) / 32), (unsigned)jobs->count), 32, b2, s>>>(*jobs);
  jobs->count = 0;
  return cudaGetLastError();
}

}  // namespace te

using namespace te;

extern "C" te_status t_mp2_bno_batched(te_handle hh, const te_mp2_cluster* cs, const te_mp2_out* outs, int64_t n,
                                       te_precision p, te_stream_t ss) {
  Handle* h = reinterpret_cast<Handle*>(hh);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(ss);
  if (!h) return fail(TE_EINVAL, "null handle");
  if (n < 0) return fail(TE_EINVAL, "negative batch size");
  if (n == 0) return TE_OK;
  if (!cs || !outs) return fail(TE_EINVAL, "null cluster or output array");
  if (p != TE_FP64 && p != TE_OZAKI)
    return fail(TE_EUNSUPPORTED, "the MP2 step runs in TE_FP64 or TE_OZAKI (got %d)", (int)p);
  if (h->capturing) return fail(TE_EINVAL, "the MP2 step cannot run inside the library's graph capture");
  if (p == TE_OZAKI && h->cc_major != 10 && h->cc_major != 11)
    return fail(TE_EUNSUPPORTED, "exact-slice contractions need an sm_100-family GPU");
  const bool oz = p == TE_OZAKI;
  size_t need_tr = 0, need_keep = 0, group_keep = 0, group_tri = 0;
  for (int64_t x = 0; x < n; ++x) {  // every descriptor before any launch
    const te_mp2_cluster& c = cs[x];
    if (c.nocc < 1 || c.nvir < 1 || c.naux < 1)
      return fail(TE_EINVAL, "cluster %lld: nocc, nvir and naux must be >= 1", (long long)x);
    if (c.nocc > 2048 || c.nvir > 4094 || c.naux > (1LL << 20))
      return fail(TE_EUNSUPPORTED, "cluster %lld too large (nocc <= 2048, nvir <= 4094)", (long long)x);
    if (!c.eps_o || !c.eps_v || !c.Bov) return fail(TE_EINVAL, "cluster %lld: null input pointer", (long long)x);
    const te_mp2_out& q = outs[x];
    if (!q.t2 && !q.gamma_oo && !q.gamma_vv && !q.pop_o && !q.pop_v)
      return fail(TE_EINVAL, "cluster %lld: no output requested", (long long)x);
    need_tr = std::max(need_tr, mp2_bytes(c.nocc, c.nvir, c.naux, oz));
    if (x % kMp2Group == 0) group_keep = group_tri = 0;
    group_tri += mp2_tri_bytes(c.nocc, c.nvir);
    need_tr = std::max(need_tr, group_tri);
    group_keep += mp2_keep_bytes(c.nocc, c.nvir);
    need_keep = std::max(need_keep, group_keep);
  }
  const size_t need = need_keep + need_tr + 1024;
  int prev = -1;
  cudaGetDevice(&prev);
  if (prev != h->device) cudaSetDevice(h->device);
  struct Restore {
    int prev, dev;
    ~Restore() {
      if (prev >= 0 && prev != dev) cudaSetDevice(prev);
    }
  } restore{prev, h->device};
  te_status st = ensure_workspace_public(h, need);
  if (st != TE_OK) return st;
  const std::unique_ptr<EigJobs> owned(new (std::nothrow) EigJobs{});
  EigJobs* const jobs = owned.get();
  if (!jobs) return fail(TE_ENOMEM, "eigensolver tables");
  cudaError_t e = cudaSuccess;
  char* const ws0 = reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(h->ws) + 255) & ~uintptr_t(255));
  char* keep = ws0;                       // kept blocks of the current group
  char* const transient = ws0 + need_keep;  // one cluster's contractions, then
  char* tri = transient;                    // the group's tridiagonal forms
  for (int64_t x = 0; x < n && e == cudaSuccess; ++x) {
    const te_mp2_cluster& c = cs[x];
    const te_mp2_out& q = outs[x];
    const int64_t o = c.nocc, v = c.nvir, P = c.naux;
    const int64_t ov = o * v, t2n = o * o * v * v;
    if (x % kMp2Group == 0) {
      keep = ws0;
      tri = transient;
    }
    auto take_from = [](char*& base, size_t bytes) {
      char* r = base;
      base += al256(bytes);
      return r;
    };
    char* base = transient;
    auto take = [&](size_t bytes) { return take_from(base, bytes); };
    double* ovov = reinterpret_cast<double*>(take((size_t)ov * ov * 8));
    double* t2 = reinterpret_cast<double*>(take((size_t)t2n * 8));
    double* tt = reinterpret_cast<double*>(take((size_t)t2n * 8));
    double* goo = reinterpret_cast<double*>(take_from(keep, (size_t)o * o * 8));
    double* gvv = reinterpret_cast<double*>(take_from(keep, (size_t)v * v * 8));
    double* eo_tri = reinterpret_cast<double*>(take_from(tri, (size_t)o * 16));
    double* ev_tri = reinterpret_cast<double*>(take_from(tri, (size_t)v * 16));
    double* eo_work = o > kEigSmemN ? reinterpret_cast<double*>(take_from(keep, (size_t)o * o * 8)) : nullptr;
    double* ev_work = v > kEigSmemN ? reinterpret_cast<double*>(take_from(keep, (size_t)v * v * 8)) : nullptr;
    const int64_t cap = mp2_scratch(o, v);
    double* scratch = reinterpret_cast<double*>(take(mp2_shared_bytes(o, v, P, oz)));
    if (q.t2) t2 = q.t2;
    if (q.gamma_oo) goo = q.gamma_oo;
    if (q.gamma_vv) gvv = q.gamma_vv;
    // input values: finite, max eps_o < min eps_v (reported by te_sync); the
    // same pass finds max |Bov|, the scale of its slices
    __nv_bfloat16* bs = reinterpret_cast<__nv_bfloat16*>(scratch);
    unsigned int* mx = oz ? reinterpret_cast<unsigned int*>(take(64)) : nullptr;
    if (oz) e = cudaMemsetAsync(mx, 0, 4, s);
    if (e == cudaSuccess)
      e = launch_check_mp2(c.eps_o, o, c.eps_v, v, c.Bov, P * ov, x, h->d_err, h->num_sms, s, mx);
    ++h->n_launches;
    // (ia|jb) = sum_P B[P,i,a] B[P,j,b]: rows (i,a), columns (j,b), K = P
    if (!oz) {
      if (e == cudaSuccess) e = cudaMemsetAsync(ovov, 0, (size_t)ov * ov * 8, s);
      if (e == cudaSuccess)
        e = gemm_strided(GemmView{c.Bov, c.Bov, ovov, o, v, ov, P, 1, v, 1, ov, 0, ov, 0, 1, v * ov, ov, 1, 1.0, true},
                         h->num_sms, scratch, cap, s, &h->n_launches);
    } else {
      int* ex = reinterpret_cast<int*>(mx + 3);
      const int64_t Pp = mp2_pitch(P);
      if (e == cudaSuccess) e = slice_rows(c.Bov, ov, P, Pp, 4, mx, ex, bs, s, &h->n_launches);
      if (e == cudaSuccess) {
        st = vt_product(h, bs, ov * Pp, ov, bs, ov * Pp, ov, P, Pp, 4, ex, ex, ovov, s);
        if (st != TE_OK) return st;
      }
    }
    // amplitudes, then the two density contractions in float64 in both modes:
    // their K (o^2 v and o v^2 terms) spans the amplitudes' whole dynamic
    // range, which one power-of-two scale per array would not resolve
    {
      if (e == cudaSuccess) {
        k_mp2_amplitudes<<<grid_of(t2n), 256, 0, s>>>(ovov, c.eps_o, c.eps_v, (int)o, (int)v, t2, tt);
        ++h->n_launches;
        e = cudaGetLastError();
      }
      if (e == cudaSuccess) e = cudaMemsetAsync(gvv, 0, (size_t)v * v * 8, s);
      if (e == cudaSuccess)
        e = gemm_strided(GemmView{t2, tt, gvv, v, 1, v, o * o, v, v, 0, v * v, 1, v * v, 1, v, v, 0, 1, 2.0},
                         h->num_sms, scratch, cap, s, &h->n_launches);
      if (e == cudaSuccess) {
        k_two_identity<<<grid_of(o * o), 256, 0, s>>>(goo, (int)o);
        ++h->n_launches;
        e = cudaGetLastError();
      }
      if (e == cudaSuccess)
        e = gemm_strided(
            GemmView{t2, tt, goo, o, 1, o, o, v * v, o * v * v, 0, v * v, 1, v * v, 1, o * v * v, o, 0, 1, -2.0},
            h->num_sms, scratch, cap, s, &h->n_launches);
    }
    // populations: the eigensolver's two launches once per group of clusters (their blocks stay in the kept region)
    if (e == cudaSuccess) {
      if (q.pop_o) jobs->j[jobs->count++] = EigJob{eo_work, goo, q.pop_o, eo_tri, eo_tri + o, (int)o};
      if (q.pop_v) jobs->j[jobs->count++] = EigJob{ev_work, gvv, q.pop_v, ev_tri, ev_tri + v, (int)v};
      if (jobs->count > 0 && ((x + 1) % kMp2Group == 0 || x + 1 == n)) {
        e = launch_eig(jobs, s);
        h->n_launches += 2;
      }
    }
  }
  if (e != cudaSuccess) return fail(TE_ECUDA, "MP2 step launch: %s", cudaGetErrorString(e));
  return TE_OK;
}
