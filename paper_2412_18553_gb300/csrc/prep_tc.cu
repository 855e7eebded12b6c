// Operand preparation of the tensor-core modes: largest magnitudes and splits.
//
// GB300 runs float64 at 2 lanes per SM and cycle, 1/64 of its FP32 and integer
// rate, so these passes over the inputs keep float64 arithmetic out: a slice
// is cut from the bits of the value by 32-bit integer operations, and a
// largest magnitude is an integer maximum over the high words.
#include <algorithm>

#include "adjoint_tc.cuh"
#include "prep_tc.h"
#include "strided.h"

namespace te {

namespace {

// ---------------------------------------------------------------------------
// one value -> the bit patterns of its parts
// ---------------------------------------------------------------------------

// Round x to the nearest value with `bits` significant bits (Veltkamp split).
// __dmul_rn / __dsub_rn keep the compiler from contracting into an FMA.
template <int BITS>
__device__ __forceinline__ double round_sig(double x) {
  const double c = __dmul_rn(x, (double)((1ull << (53 - BITS)) + 1ull));
  return __dsub_rn(c, __dsub_rn(c, x));
}

__device__ __forceinline__ uint32_t bf16_bits(double x) {  // x exact in BF16
  return __float_as_uint((float)x) >> 16;
}

// The slices m_k of t = x 2^-e, |t| < 1, by repeated rounding to nearest even:
// t 2^beta = m_0 + r_0, r_0 2^beta = m_1 + r_1, ...  |t| 2^32 as a 32-bit
// integer whose lowest bit also says whether anything was cut off below it;
// every rounding threshold is an even integer, so each comparison comes out as
// on the exact value.  |t| below 2^-1022 counts as zero.
template <int BETA, int NS>
__device__ __forceinline__ void rint_digits(double x, int e, int* m) {
  static_assert(32 - BETA * NS >= 2, "the last threshold is an even integer");
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const int E = (int)((hi >> 20) & 0x7FFu);
  const uint32_t mant = 0x80000000u | ((hi & 0xFFFFFu) << 11) | (lo >> 21);  // 1.f at bit 31
  const uint32_t sh = (uint32_t)(e + 1022 - E);  // |x| < 2^e: not negative
  uint32_t A = 0, rest = lo & 0x1FFFFFu;
  if (sh < 32u) {
    A = mant >> sh;
    rest |= mant & ((1u << sh) - 1u);
  } else {
    rest = 1u;
  }
  A = E == 0 ? 0u : (A | (rest ? 1u : 0u));
  constexpr int P0 = 32 - BETA;
  uint32_t q = A >> P0;
  {
    const uint32_t rem = A & ((1u << P0) - 1u), half = 1u << (P0 - 1);
    q += (rem > half || (rem == half && (q & 1u))) ? 1u : 0u;
  }
  const int sgn = (int)hi >> 31;  // 0 or -1
  m[0] = ((int)q ^ sgn) - sgn;
  int r = (int)(A - (q << P0));
#pragma unroll
  for (int k = 1; k < NS; ++k) {
    const int P = 32 - BETA * (k + 1);
    int d = r >> P;
    const int rem = r & ((1 << P) - 1), half = 1 << (P - 1);
    d += (rem > half || (rem == half && (d & 1))) ? 1 : 0;
    r -= d << P;
    m[k] = (d ^ sgn) - sgn;
  }
}

// the bit patterns of x's parts
template <int MODE>
__device__ __forceinline__ void split_value(double x, int e, uint32_t* w) {
  constexpr int NS = ModeTraits<MODE>::nparts;
  if constexpr (MODE == TC_OZAKI || MODE == TC_OZAKI6) {
    constexpr int BETA = ModeTraits<MODE>::beta;
    int m[NS];
    rint_digits<BETA, NS>(x, e, m);
#pragma unroll
    for (int k = 0; k < NS; ++k) w[k] = digit_bf16(m[k], BETA * (k + 1));
  } else if constexpr (MODE == TC_SLICE4 || MODE == TC_SLICE5) {
    int d[NS];
    slice_digits_int<NS>(x, e, d);
#pragma unroll
    for (int k = 0; k < NS; ++k) w[k] = digit_bf16(d[k], 7 * (k + 1));
  } else if constexpr (MODE == TC_BF16X3) {
    const double h = round_sig<8>(x);
    w[0] = bf16_bits(h);
    w[1] = bf16_bits(round_sig<8>(x - h));
  } else {
    const double h = round_sig<11>(x);
    w[0] = __float_as_uint((float)h);
    if constexpr (MODE == TC_TF32X3) w[1] = __float_as_uint((float)round_sig<11>(x - h));
  }
}

// entries of the energy modes' scale table from max |ovvv|, |t2|, |ooov|
__device__ __forceinline__ int energy_exp(const unsigned int* maxhi, int which) {
  const int ev = exp_of_high(maxhi[0]), et = exp_of_high(maxhi[1]), eo = exp_of_high(maxhi[2]);
  const int U = max(ev + et, et + eo);
  return which == 0 ? U - et : (which == 1 ? et : (which == 2 ? U - eo : (which == 3 ? eo : U)));
}

struct SplitLaunch {
  SplitJob job[SPLIT_MAX_JOBS];
  int njobs;
  SplitScales sc;
};

constexpr int SPLIT_THREADS = 256;
constexpr int SPLIT_CHUNKS = 4;  // chunks of four elements per thread (rows)

__device__ __forceinline__ int row_exp(const SplitJob& J, const SplitScales& sc, uint32_t group) {
  if (J.gexp) return exp_of_high(sc.group_hi[(J.gexp - sc.group_exps) + group]);
  return sc.maxhi ? energy_exp(sc.maxhi, J.which) : 0;
}

// Four consecutive elements per chunk: 32 bytes read and 4 es bytes written
// per part and lane, so that a warp's accesses are whole lines on both sides.
// All of a thread's loads are issued before the first conversion.
template <int MODE>
__device__ __forceinline__ void split_rows(const SplitJob& J, const SplitScales& sc, int64_t blk) {
  constexpr int NS = ModeTraits<MODE>::nparts, ES = ModeTraits<MODE>::es;
  const uint32_t cpr = (uint32_t)J.Kp / 4u;
  const int64_t total = J.n * cpr, base = blk * (SPLIT_THREADS * SPLIT_CHUNKS);
  const int64_t row0 = base / cpr;
  const uint32_t col0 = (uint32_t)(base - row0 * cpr);
  const bool vec = (J.K & 1) == 0 && (reinterpret_cast<uintptr_t>(J.src) & 15) == 0;
  double x[SPLIT_CHUNKS][4];
  uint32_t row[SPLIT_CHUNKS], col[SPLIT_CHUNKS];
#pragma unroll
  for (int i = 0; i < SPLIT_CHUNKS; ++i) {
    const uint32_t l = col0 + i * SPLIT_THREADS + threadIdx.x;
    const uint32_t dr = l / cpr;
    row[i] = (uint32_t)row0 + dr;
    col[i] = (l - dr * cpr) * 4u;
    const bool live = base + i * SPLIT_THREADS + threadIdx.x < total;
    const double* s = J.src + (int64_t)row[i] * J.K + col[i];
    if (live && vec && (int)col[i] + 4 <= J.K) {
      const double2 a = __ldg(reinterpret_cast<const double2*>(s)), b = __ldg(reinterpret_cast<const double2*>(s) + 1);
      x[i][0] = a.x;
      x[i][1] = a.y;
      x[i][2] = b.x;
      x[i][3] = b.y;
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) x[i][j] = (live && (int)col[i] + j < J.K) ? __ldg(s + j) : 0.0;
    }
  }
#pragma unroll
  for (int i = 0; i < SPLIT_CHUNKS; ++i) {
    if (base + i * SPLIT_THREADS + threadIdx.x >= total) break;
    const uint32_t G = (uint32_t)J.G, g = row[i] / G, rin = row[i] - g * G;
    const int e = row_exp(J, sc, g);
    uint32_t w[4][NS];
#pragma unroll
    for (int j = 0; j < 4; ++j) split_value<MODE>(x[i][j], e, w[j]);
    const int64_t at = (int64_t)g * ((int64_t)NS * J.G * J.Kp) + (int64_t)rin * J.Kp + col[i];
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      char* d = static_cast<char*>(J.parts.p[k]) + at * ES;
      if constexpr (ES == 2)
        *reinterpret_cast<uint2*>(d) = make_uint2(__byte_perm(w[0][k], w[1][k], 0x5410), __byte_perm(w[2][k], w[3][k], 0x5410));
      else
        *reinterpret_cast<uint4*>(d) = make_uint4(w[0][k], w[1][k], w[2][k], w[3][k]);
    }
  }
}

// A thread takes eight consecutive l of one output row: its eight loads are
// each contiguous over the warp (lanes along i), its store is 8 es bytes per
// part; neighbouring blocks of l are the next threads' and fill the line.
template <int MODE>
__device__ __forceinline__ void split_cols(const SplitJob& J, const SplitScales& sc, int64_t blk) {
  constexpr int NS = ModeTraits<MODE>::nparts, ES = ModeTraits<MODE>::es;
  const int64_t rows = J.n * J.nb, lane = blk * SPLIT_THREADS + threadIdx.x;
  if (lane >= rows) return;
  const uint32_t r = (uint32_t)lane, n = (uint32_t)J.n, b = r / n, i = r - b * n;
  const uint32_t G = (uint32_t)J.G, g = r / G, rin = r - g * G;
  const int e = row_exp(J, sc, g);
  const double* s = J.src + (int64_t)b * J.bs + i;
  const int64_t at0 = (int64_t)g * ((int64_t)NS * J.G * J.Kp) + (int64_t)rin * J.Kp;
  for (int l0 = 0; l0 < J.Kp; l0 += 8) {
    double x[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) x[j] = l0 + j < J.K ? __ldg(s + (int64_t)(l0 + j) * J.ls) : 0.0;
    uint32_t p[NS][8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      uint32_t w[NS];
      split_value<MODE>(J.sign < 0 ? -x[j] : x[j], e, w);
#pragma unroll
      for (int k = 0; k < NS; ++k) p[k][j] = w[k];
    }
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      char* d = static_cast<char*>(J.parts.p[k]) + (at0 + l0) * ES;
      if constexpr (ES == 2) {
        uint32_t q[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) q[j] = __byte_perm(p[k][2 * j], p[k][2 * j + 1], 0x5410);
        *reinterpret_cast<uint4*>(d) = make_uint4(q[0], q[1], q[2], q[3]);
      } else {
        *reinterpret_cast<uint4*>(d) = make_uint4(p[k][0], p[k][1], p[k][2], p[k][3]);
        *(reinterpret_cast<uint4*>(d) + 1) = make_uint4(p[k][4], p[k][5], p[k][6], p[k][7]);
      }
    }
  }
}

// K = v, Kp = vq, n = o: element (i, a, j, b) of the float32 symmetrised ovov
__device__ __forceinline__ void split_ovs(const SplitJob& J, int64_t blk) {
  const int o = (int)J.n, v = J.K, vq = J.Kp;
  const int64_t total = (int64_t)o * v * o * vq;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int64_t idx = blk * (4 * SPLIT_THREADS) + u * SPLIT_THREADS + threadIdx.x;
    if (idx >= total) return;
    const int64_t row = idx / vq;  // (i v + a) o + j
    const int b = (int)(idx - row * vq);
    const uint32_t r = (uint32_t)row, ia = r / (uint32_t)o, j = r - ia * (uint32_t)o;
    const uint32_t i = ia / (uint32_t)v, a = ia - i * (uint32_t)v;
    float val = 0.f;
    if (b < v)
      val = (float)(0.5 * (J.src[(int64_t)row * v + b] + J.src[(((int64_t)j * v + b) * o + i) * v + a]));
    J.dst32[idx] = val;
  }
}

__device__ __forceinline__ void split_copy(const SplitJob& J, int64_t blk) {
  const int64_t idx = blk * SPLIT_THREADS + threadIdx.x, total = J.n * J.Kp;
  if (idx >= total) return;
  const int64_t row = idx / J.Kp;
  const int k = (int)(idx - row * J.Kp);
  J.dst32[idx] = k < J.K ? (float)J.src[row * J.K + k] : 0.f;
}

int64_t split_blocks(const SplitJob& J) {
  const int64_t T = SPLIT_THREADS;
  switch (J.kind) {
    case SPLIT_ROWS: return (J.n * (J.Kp / 4) + T * SPLIT_CHUNKS - 1) / (T * SPLIT_CHUNKS);
    case SPLIT_COLS: return (J.n * J.nb + T - 1) / T;
    case SPLIT_OVS: return (J.n * J.K * J.n * J.Kp + 4 * T - 1) / (4 * T);
    default: return (J.n * J.Kp + T - 1) / T;
  }
}

// Every split of a call in one launch: a block belongs to one job.  HBM bounds
// it in the end (8 bytes read and 2 NS written per element: 2.7 ms for all
// operands of nocc=32 nvir=320, 18 GB), the integer instructions come next.
// Measured there, four 7-bit slices: 5.2 ms, against 45.6 ms for separate
// kernels that rounded in float64 (seventeen float64 operations per element on
// two lanes per SM and cycle) and read t2L's source across its rows.
template <int MODE>
__global__ void __launch_bounds__(SPLIT_THREADS) k_split(const __grid_constant__ SplitLaunch L) {
  int j = 0;
  while (j + 1 < L.njobs && L.job[j + 1].block0 <= (int64_t)blockIdx.x) ++j;
  const SplitJob& J = L.job[j];
  const int64_t blk = (int64_t)blockIdx.x - J.block0;
  if (blockIdx.x == 0) {
    if (L.sc.maxhi && threadIdx.x < 5) L.sc.exps[threadIdx.x] = energy_exp(L.sc.maxhi, (int)threadIdx.x);
    for (int g = threadIdx.x; g < L.sc.ngroups; g += SPLIT_THREADS) L.sc.group_exps[g] = exp_of_high(L.sc.group_hi[g]);
  }
  if (J.kind == SPLIT_ROWS) split_rows<MODE>(J, L.sc, blk);
  else if (J.kind == SPLIT_COLS) split_cols<MODE>(J, L.sc, blk);
  else if (J.kind == SPLIT_OVS) split_ovs(J, blk);
  else split_copy(J, blk);
}

// ---------------------------------------------------------------------------
// largest magnitudes and the finite check
// ---------------------------------------------------------------------------

struct MaxLaunch {
  MaxArray a[MAX_ARRAYS];
  int64_t task0[MAX_ARRAYS], ntasks;
  int cpr[MAX_ARRAYS];  // chunks per row
  int n;
  const double *eps_o, *eps_v;
  int o, v;
  unsigned int cluster;
};

constexpr int MAX_CHUNK = 4096;  // entries per warp task

__device__ __forceinline__ void report(unsigned int* err, unsigned int site, unsigned int cluster) {
  if (atomicOr(err, ERR_BAD_INPUT) == 0) {
    err[1] = site;
    err[2] = cluster;
  }
}

// A warp takes a run of at most MAX_CHUNK entries of one row: eight 16-byte
// loads in flight per lane, then one integer maximum per entry.  HBM bounds it:
// 1.40 ms for the 9 GB of nocc=32 nvir=320 (6.4 TB/s), where a check pass and a
// float64 fmax pass took 1.55 + 2.35 ms.
__device__ __forceinline__ unsigned int warp_max(const double* p, int64_t n, int lane) {
  unsigned int m = 0;
  if (n > 0 && (reinterpret_cast<uintptr_t>(p) & 8)) {  // up to a 16-byte boundary
    if (lane == 0) m = (unsigned int)__double2hiint(__ldg(p)) & 0x7FFFFFFFu;
    ++p;
    --n;
  }
  const uint4* q = reinterpret_cast<const uint4*>(p);
  const int n2 = (int)(n >> 1);
  int i = lane;
  for (; i + 7 * 32 < n2; i += 8 * 32) {
    uint4 w[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) w[u] = __ldg(q + i + u * 32);
#pragma unroll
    for (int u = 0; u < 8; ++u) m = max(m, max(w[u].y & 0x7FFFFFFFu, w[u].w & 0x7FFFFFFFu));
  }
  for (; i < n2; i += 32) {
    const uint4 w = __ldg(q + i);
    m = max(m, max(w.y & 0x7FFFFFFFu, w.w & 0x7FFFFFFFu));
  }
  if ((n & 1) && lane == 0) m = max(m, (unsigned int)__double2hiint(__ldg(p + n - 1)) & 0x7FFFFFFFu);
  return __reduce_max_sync(0xffffffffu, m);
}

__global__ void __launch_bounds__(256) k_absmax(const __grid_constant__ MaxLaunch L, unsigned int* err) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int64_t t = blockIdx.x * 8LL + warp; t < L.ntasks; t += gridDim.x * 8LL) {
    int w = 0;
    while (w + 1 < L.n && L.task0[w + 1] <= t) ++w;
    const MaxArray& A = L.a[w];
    const int64_t lt = t - L.task0[w], row = lt / L.cpr[w];
    const int64_t c0 = (lt - row * L.cpr[w]) * MAX_CHUNK;
    const unsigned int m = warp_max(A.p + row * A.len + c0, min((int64_t)MAX_CHUNK, A.len - c0), lane);
    if (lane == 0) {
      if (A.out) {
        const int64_t g = A.o == 0 ? 0 : (A.o < 0 ? row : (row / ((int64_t)A.o * A.o)) * A.o + row % A.o);
        if (m > *(volatile unsigned int*)(A.out + g)) atomicMax(A.out + g, m);
      }
      if (A.out2 && m > *(volatile unsigned int*)(A.out2 + row % A.o2)) atomicMax(A.out2 + row % A.o2, m);
      if (m >= 0x7FF00000u && A.site) report(err, A.site, L.cluster);
    }
  }
  if (blockIdx.x == 0 && L.eps_o) {  // max(eps_o) < min(eps_v)
    __shared__ double smax[8], smin[8];
    double mo = -1.0e308, mv = 1.0e308;
    for (int i = threadIdx.x; i < L.o; i += blockDim.x) mo = fmax(mo, L.eps_o[i]);
    for (int i = threadIdx.x; i < L.v; i += blockDim.x) mv = fmin(mv, L.eps_v[i]);
    for (int off = 16; off > 0; off >>= 1) {
      mo = fmax(mo, __shfl_down_sync(0xffffffffu, mo, off));
      mv = fmin(mv, __shfl_down_sync(0xffffffffu, mv, off));
    }
    if (lane == 0) {
      smax[warp] = mo;
      smin[warp] = mv;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
        mo = fmax(mo, smax[w]);
        mv = fmin(mv, smin[w]);
      }
      if (!(mo < mv)) report(err, 8u, L.cluster);
    }
  }
}

// NS 7-bit slices of x[0..n) by repeated rounding to nearest even, as
// rint_digits, from a 48-bit integer (NS = 5 needs 35 bits and the rounding
// bits below them)
template <int NS>
__device__ __forceinline__ void rint_digits_wide(double x, int e, int* m) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const int E = (int)((bits >> 52) & 0x7FFull);
  const unsigned long long M = (bits & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const unsigned int sh = (unsigned int)(1027 + e - E);  // |x| 2^(48 - e) = M 2^-sh; |x| < 2^e: at least 5
  unsigned long long A = 1ull;
  if (sh < 64u) A = (M >> sh) | ((M & ((1ull << sh) - 1ull)) ? 1ull : 0ull);
  if (E == 0) A = 0;
  long long r = (long long)A;
  const int sgn = (int)(bits >> 63) ? -1 : 0;
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const int P = 48 - 7 * (k + 1);
    int d = (int)(r >> P);
    const long long rem = r & ((1ll << P) - 1ll), half = 1ll << (P - 1);
    d += (rem > half || (rem == half && (d & 1))) ? 1 : 0;
    r -= (long long)d << P;
    m[k] = (d ^ sgn) - sgn;
  }
}

// x [P][n] to rows of K: slice s of x[p][i] at planes[(s n + i) Pp + p], the
// K-contiguous rows that a tensor map reads.  A block takes 64 p x 32 i: x is read
// along i, the planes are written along p (128 bytes per row and slice).
constexpr int SP_P = 64, SP_I = 32;
template <int NS>
__global__ void __launch_bounds__(256) k_slice_rows(const double* __restrict__ x, int64_t n, int64_t P, int64_t Pp,
                                                    const unsigned int* __restrict__ xhi, int* __restrict__ e_out,
                                                    unsigned short* __restrict__ planes) {
  __shared__ unsigned short t[NS][SP_I][SP_P + 2];
  const int e = exp_of_high(*xhi), tid = threadIdx.x;
  if (blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) *e_out = e;
  const int64_t i0 = (int64_t)blockIdx.x * SP_I, p0 = (int64_t)blockIdx.y * SP_P;
#pragma unroll
  for (int q = tid; q < SP_P * SP_I; q += 256) {
    const int i = q % SP_I, p = q / SP_I;
    int d[NS];
    rint_digits_wide<NS>(i0 + i < n && p0 + p < P ? __ldg(x + (p0 + p) * n + i0 + i) : 0.0, e, d);
#pragma unroll
    for (int k = 0; k < NS; ++k) t[k][i][p] = (unsigned short)digit_bf16(d[k], 7 * (k + 1));
  }
  __syncthreads();
  for (int q = tid; q < NS * SP_I * (SP_P / 2); q += 256) {
    const int p = 2 * (q % (SP_P / 2)), r = q / (SP_P / 2), i = r % SP_I, k = r / SP_I;
    if (i0 + i < n && p0 + p < Pp)  // Pp is even
      *reinterpret_cast<uint32_t*>(planes + ((int64_t)k * n + i0 + i) * Pp + p0 + p) =
          *reinterpret_cast<const uint32_t*>(&t[k][i][p]);
  }
}

}  // namespace

cudaError_t slice_rows(const double* x, int64_t n, int64_t P, int64_t Pp, int ns, const unsigned int* xhi, int* ex,
                       __nv_bfloat16* planes, cudaStream_t s, int64_t* launches) {
  if ((ns != 4 && ns != 5) || P > 65535LL * SP_P || n > 0x7FFFFFFFLL) return cudaErrorInvalidValue;
  const dim3 grid((unsigned)((n + SP_I - 1) / SP_I), (unsigned)((P + SP_P - 1) / SP_P));
  unsigned short* p = reinterpret_cast<unsigned short*>(planes);
  if (ns == 5) k_slice_rows<5><<<grid, 256, 0, s>>>(x, n, P, Pp, xhi, ex, p);
  else k_slice_rows<4><<<grid, 256, 0, s>>>(x, n, P, Pp, xhi, ex, p);
  ++*launches;
  return cudaGetLastError();
}

cudaError_t launch_split(int mode, const SplitJob* jobs, int njobs, const SplitScales& sc, cudaStream_t s) {
  if (njobs < 1 || njobs > SPLIT_MAX_JOBS) return cudaErrorInvalidValue;
  SplitLaunch L{};
  int64_t blocks = 0;
  for (int q = 0; q < njobs; ++q) {
    L.job[q] = jobs[q];
    L.job[q].block0 = blocks;
    blocks += split_blocks(jobs[q]);
  }
  L.njobs = njobs;
  L.sc = sc;
  if (blocks > 0x7FFFFFFF) return cudaErrorInvalidValue;
  const unsigned g = (unsigned)std::max<int64_t>(1, blocks);
  switch (mode) {
    case TC_BF16X3: k_split<TC_BF16X3><<<g, SPLIT_THREADS, 0, s>>>(L); break;
    case TC_TF32X3: k_split<TC_TF32X3><<<g, SPLIT_THREADS, 0, s>>>(L); break;
    case TC_TF32: k_split<TC_TF32><<<g, SPLIT_THREADS, 0, s>>>(L); break;
    case TC_OZAKI: k_split<TC_OZAKI><<<g, SPLIT_THREADS, 0, s>>>(L); break;
    case TC_OZAKI6: k_split<TC_OZAKI6><<<g, SPLIT_THREADS, 0, s>>>(L); break;
    case TC_SLICE4: k_split<TC_SLICE4><<<g, SPLIT_THREADS, 0, s>>>(L); break;
    case TC_SLICE5: k_split<TC_SLICE5><<<g, SPLIT_THREADS, 0, s>>>(L); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_absmax(const MaxArray* arrays, int n, const double* eps_o, int o, const double* eps_v, int v,
                          unsigned int cluster, unsigned int* err, int num_sms, cudaStream_t s) {
  if (n < 0 || n > MAX_ARRAYS) return cudaErrorInvalidValue;
  MaxLaunch L{};
  for (int q = 0; q < n; ++q) {
    if (arrays[q].rows <= 0 || arrays[q].len <= 0) continue;
    const int k = L.n++;
    L.a[k] = arrays[q];
    L.cpr[k] = (int)((arrays[q].len + MAX_CHUNK - 1) / MAX_CHUNK);
    L.task0[k] = L.ntasks;
    L.ntasks += arrays[q].rows * L.cpr[k];
  }
  L.eps_o = eps_o;
  L.eps_v = eps_v;
  L.o = o;
  L.v = v;
  L.cluster = cluster;
  const int64_t grid = std::max<int64_t>(1, std::min<int64_t>((L.ntasks + 7) / 8, 8LL * std::max(1, num_sms)));
  k_absmax<<<(unsigned)grid, 256, 0, s>>>(L, err);
  return cudaGetLastError();
}

}  // namespace te
