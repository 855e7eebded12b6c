// The exact-slice adjoint of E(T) (see vjp.cu for the formulas): contractions on
// tcgen05 (view_tc.cu), everything else in float64.
//
// Triples go in batches of consecutive canonical triples (up to eight, as many
// as about a gigabyte of G, dW~ and layouts holds), and each stage is one launch
// over the batch: at nocc=16 nvir=120 a triple's stages are 10 to 100 us each,
// and launched triple by triple their tails and launch gaps cost as much as
// their work.  Contributions of a batch to one output block are segments of one
// job, in triple order, so every accumulation has a fixed order.
//
// What bounds the kernels around the contractions, one triple at nvir = 320: the
// epilogue (1.27 ms; a warp along one orbit index, whose G reads touch 32 lines,
// 1.85; 4 v^3 values moved would take 0.16) and the Y and denominator planes (0.65) their
// float64 operations, about 106 per orbit and 8 per value at two lanes per SM and
// cycle; the dW~ slices (0.55 ms for all six layouts, cut once; 1.01 when cut for three
// at a time) memory.  The view GEMM launches take 5.6 of the 9.2 ms (view_tc.cu).
//
// Where the operand transposes of all occupied indices would take too much
// memory (a large cluster: full = false) a triple goes alone, the transposes are
// made when they are due and the dW~ layouts come three at a time.
#include <cuda_bf16.h>

#include <algorithm>
#include <initializer_list>
#include <map>
#include <new>
#include <vector>

#include "adjoint_tc.cuh"
#include "prep_tc.h"
#include "strided.h"
#include "tc_path.h"
#include "te_internal.h"
#include "view_tc.h"

namespace te {

te_status ensure_triples_public(Handle* h, int nocc);

namespace {

using bf = __nv_bfloat16;

constexpr int ADJ_MAX_BATCH = 8;
constexpr int64_t ADJ_BATCH_BYTES = int64_t(1) << 30;   // G, dW~ and layouts of a batch
constexpr int64_t ADJ_FULL_BYTES = int64_t(12) << 30;   // most extra workspace for the transposes of all indices

// ---------------------------------------------------------------------------
// epilogue
// ---------------------------------------------------------------------------

struct AdjBatch {
  int n;             // triples (slots) of the batch
  Triple t[ADJ_MAX_BATCH];
  double w[ADJ_MAX_BATCH];  // gE m / 3
};

struct AdjEpi {
  AdjArgs a;          // inputs; G of slot 0
  double* dW;         // [slot][v^3]
  double *dY, *dD;    // [slot][v^3]
  int64_t g_stride, d_stride, w_stride;  // doubles per slot of G; of dY and dD; of dW
  unsigned long long* dwmax;  // [slot] bits of max |dW|
  double *epart, *dpart;  // [slot][gridDim.x] sums of the share (m / 3 apart) and of dD
};

// Threads stride over the orbits a >= b >= c (v(v+1)(v+2)/6 of them): W~ and Y
// are formed once per orbit and every distinct element of the orbit gets its
// dW~, dY and dD.  1/D: two Newton steps from an FP32 seed.
__global__ void __launch_bounds__(256) k_adjoint_batch(const __grid_constant__ AdjEpi A,
                                                       const __grid_constant__ AdjBatch B) {
  __shared__ double red[8], redd[8], redw[8];
  const int slot = blockIdx.y;
  const Triple T = B.t[slot];
  AdjArgs a = A.a;
  a.G += slot * A.g_stride;
  a.i = T.i;
  a.j = T.j;
  a.k = T.k;
  const double w = B.w[slot];
  const int64_t v = a.v, steps = orbit_steps(a.v);
  const OrbitTile tile = orbit_tile();
  double* dW = A.dW + slot * A.w_stride;
  double* dY = A.dY + slot * A.d_stride;
  double* dD = A.dD + slot * A.d_stride;
  const double eo = a.eps_o[T.i] + a.eps_o[T.j] + a.eps_o[T.k];
  double cs = 0.0, ds = 0.0, wmax = 0.0;
  for (int64_t t = blockIdx.x; t < steps; t += gridDim.x) {
    int x, y, z;
    if (!orbit_at(tile, t, (int)v, &x, &y, &z)) continue;
    double W[6], Y[6], RW[6], RY[6];
    int64_t idx[6];
    orbit_values(a, x, y, z, W, Y);
    orbit_index(v, x, y, z, idx);
    r_orbit_sums(W, RW);
    r_orbit_sums(Y, RY);
    const unsigned distinct = orbit_distinct(x, y, z);
    const double D = eo - a.eps_v[x] - a.eps_v[y] - a.eps_v[z];
    const double rD = recip_newton(D, recip_newton(D, recip_seed(D)));
    const double q = w * rD;
    const double qr = -q * rD;
    double se = 0.0;  // the orbit's W~ R[V]
#pragma unroll
    for (int n = 0; n < 6; ++n) {
      if (!(distinct >> n & 1u)) continue;
      const double dw = q * fma(2.0, RW[n], RY[n]);
      dW[idx[n]] = dw;
      const unsigned long long m = (unsigned long long)__double_as_longlong(dw) & 0x7FFFFFFFFFFFFFFFull;
      if (m > (unsigned long long)__double_as_longlong(wmax)) wmax = __longlong_as_double((long long)m);
      const double e = W[n] * (RW[n] + RY[n]);
      dY[idx[n]] = q * RW[n];
      dD[idx[n]] = qr * e;
      se += e;
    }
    cs = fma(se, rD, cs);
    ds = fma(se, qr, ds);
  }
  for (int off = 16; off > 0; off >>= 1) {
    cs += __shfl_down_sync(0xffffffffu, cs, off);
    ds += __shfl_down_sync(0xffffffffu, ds, off);
    wmax = fmax(wmax, __shfl_down_sync(0xffffffffu, wmax, off));
  }
  if ((threadIdx.x & 31) == 0) {
    red[threadIdx.x >> 5] = cs;
    redd[threadIdx.x >> 5] = ds;
    redw[threadIdx.x >> 5] = wmax;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0, sd = 0.0, m = 0.0;
    for (int k = 0; k < 8; ++k) {
      s += red[k];
      sd += redd[k];
      m = fmax(m, redw[k]);
    }
    A.epart[(int64_t)slot * gridDim.x + blockIdx.x] = s;
    A.dpart[(int64_t)slot * gridDim.x + blockIdx.x] = sd;
    if (m > 0.0) atomicMax(A.dwmax + slot, (unsigned long long)__double_as_longlong(m));
  }
}

// ---------------------------------------------------------------------------
// Y and denominator reductions
// ---------------------------------------------------------------------------

// Partial results of a slot:
//   s[m] [v][v]: d ovs of mode 0 (i,a; j,b), 1 (j,b; k,c), 2 (i,a; k,c)
//   p[0], p[1] [v][v]: per first index a, the sums behind dt1 of k (at c) and of j (at b)
//   p[2], p[3] [v][v]: per a, the sums of dD behind d eps_v at b and at c
//   q[0], q[1] [v]: dt1 of i (at a), and d eps_v's sums at a
struct YParts {
  double *s[3], *p[4], *q[2];
  int64_t stride;  // doubles between slots
};

// sum over the warp, in lane 0
__device__ __forceinline__ void warp_sum(double& s) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
}

// The sums over the warp of 16 values: number i ends in the lanes l with
// l >> 1 = bits of i reversed (warp_sum16_index).  Halves are exchanged and added, so
// that 16 sums take 16 additions, not 80.
__device__ __forceinline__ double warp_sum16(double (&x)[16], int lane) {
#pragma unroll
  for (int n = 8, off = 16; n >= 1; n >>= 1, off >>= 1) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < n; ++i) {
      const double mine = up ? x[i + n] : x[i], other = up ? x[i] : x[i + n];
      x[i] = mine + __shfl_xor_sync(0xffffffffu, other, off);
    }
  }
  return x[0] + __shfl_xor_sync(0xffffffffu, x[0], 1);
}
__device__ __forceinline__ int warp_sum16_index(int lane) {
  return ((lane >> 4) & 1) * 8 + ((lane >> 3) & 1) * 4 + ((lane >> 2) & 1) * 2 + ((lane >> 1) & 1);
}

// One block per plane a of a slot: its rows (four per warp, lanes along c), then
// its columns (lanes along c, warps along b).  The plane is read twice, from L2.
__global__ void __launch_bounds__(256) k_y_planes(const __grid_constant__ AdjEpi A, const __grid_constant__ AdjBatch B,
                                                  const __grid_constant__ YParts Yp) {
  __shared__ double red[2][8];
  const int a = blockIdx.x, slot = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const Triple T = B.t[slot];
  const int v = A.a.v, o = A.a.o;
  const int64_t V = v, plane = (int64_t)a * V * V;
  const double* dY = A.dY + slot * A.d_stride + plane;
  const double* dD = A.dD + slot * A.d_stride + plane;
  const double* t1k = A.a.t1 + (int64_t)T.k * v;
  const double* t1j = A.a.t1 + (int64_t)T.j * v;
  auto ovs = [&](int p1, int x, int p2) { return A.a.ovs + (((int64_t)p1 * v + x) * o + p2) * v; };
  const double* ovs_ik = ovs(T.i, a, T.k);
  const double* ovs_ij = ovs(T.i, a, T.j);
  const int64_t so = slot * Yp.stride;
  double all = 0.0, alld = 0.0;
  for (int b0 = warp; b0 < v; b0 += 32) {  // rows b0 + 8 u
    double s[16] = {};  // [4 u + k]: sums behind d ovs of (i, j), dt1 of j and d eps_v at b
    const double* ovs_jk[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) ovs_jk[u] = ovs(T.j, min(b0 + 8 * u, v - 1), T.k);
    for (int c = lane; c < v; c += 32) {
      double y[4], d[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const bool in = b0 + 8 * u < v;
        y[u] = in ? __ldg(dY + (int64_t)(b0 + 8 * u) * V + c) : 0.0;
        d[u] = in ? __ldg(dD + (int64_t)(b0 + 8 * u) * V + c) : 0.0;
      }
      const double tk = t1k[c], oik = ovs_ik[c];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (b0 + 8 * u >= v) break;
        s[4 * u] = fma(y[u], tk, s[4 * u]);
        s[4 * u + 1] = fma(y[u], oik, s[4 * u + 1]);
        s[4 * u + 2] += d[u];
        all = fma(y[u], ovs_jk[u][c], all);
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) alld += s[4 * u + 2];
    const double t = warp_sum16(s, lane);
    const int i = warp_sum16_index(lane), b = b0 + 8 * (i >> 2), k = i & 3;
    if ((lane & 1) == 0 && k < 3 && b < v) (k == 0 ? Yp.s[0] : (k == 1 ? Yp.p[1] : Yp.p[2]))[so + a * V + b] = t;
  }
  // columns: 32 at a time, warp w takes the rows b = w, w + 8, ...
  __shared__ double col[3][8][33];
  for (int c0 = 0; c0 < v; c0 += 32) {
    const int c = c0 + lane;
    const bool in = c < v;
    double s2 = 0.0, p0 = 0.0, sd = 0.0;
    for (int b0 = warp; b0 < v; b0 += 32) {
      double y[4], d[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const bool ok = in && b0 + 8 * u < v;
        y[u] = ok ? __ldg(dY + (int64_t)(b0 + 8 * u) * V + c) : 0.0;
        d[u] = ok ? __ldg(dD + (int64_t)(b0 + 8 * u) * V + c) : 0.0;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (b0 + 8 * u >= v) break;
        s2 = fma(y[u], t1j[b0 + 8 * u], s2);
        p0 = fma(y[u], ovs_ij[b0 + 8 * u], p0);
        sd += d[u];
      }
    }
    col[0][warp][lane] = s2;
    col[1][warp][lane] = p0;
    col[2][warp][lane] = sd;
    __syncthreads();
    if (warp < 3 && in) {
      double t = 0.0;
#pragma unroll
      for (int w = 0; w < 8; ++w) t += col[warp][w][lane];
      double* out = warp == 0 ? Yp.s[2] : (warp == 1 ? Yp.p[0] : Yp.p[3]);
      out[so + a * V + c] = t;
    }
    __syncthreads();
  }
  warp_sum(all);
  warp_sum(alld);
  if (lane == 0) {
    red[0][warp] = all;
    red[1][warp] = alld;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0, td = 0.0;
    for (int w = 0; w < 8; ++w) {
      t += red[0][w];
      td += red[1][w];
    }
    Yp.q[0][so + a] = t;
    Yp.q[1][so + a] = td;
  }
}

// s[1][b][c] = sum_a dY[a,b,c] t1[i,a]
__global__ void __launch_bounds__(256) k_y_sum_a(const __grid_constant__ AdjEpi A, const __grid_constant__ AdjBatch B,
                                                 const __grid_constant__ YParts Yp) {
  const int slot = blockIdx.y, v = A.a.v;
  const int64_t v2 = (int64_t)v * v, bc = blockIdx.x * 256LL + threadIdx.x;
  if (bc >= v2) return;
  const double* dY = A.dY + slot * A.d_stride + bc;
  const double* t1i = A.a.t1 + (int64_t)B.t[slot].i * v;
  double s = 0.0;
#pragma unroll 8
  for (int a = 0; a < v; ++a) s = fma(__ldg(dY + a * v2), t1i[a], s);
  Yp.s[1][slot * Yp.stride + bc] = s;
}

// the p arrays summed over a: block (32 columns, slot, array), into rows 0 of p
__global__ void __launch_bounds__(256) k_y_columns(const __grid_constant__ YParts Yp, int v) {
  __shared__ double t[8][33];
  const int lane = threadIdx.x & 31, part = threadIdx.x >> 5, z = blockIdx.x * 32 + lane;
  double* p = Yp.p[blockIdx.z] + blockIdx.y * Yp.stride;
  double s = 0.0;
  if (z < v)
    for (int a = part; a < v; a += 8) s += p[(int64_t)a * v + z];
  t[part][lane] = s;
  __syncthreads();
  if (part == 0 && z < v) {
    for (int k = 1; k < 8; ++k) s += t[k][lane];
    p[z] = s;  // every row of this column has been read by this block
  }
}

// Outputs (nullable) and the order in which the slots' parts are added.
struct AdjOut {
  double *eps_o, *eps_v, *t1, *dOVS, *shares;
  int64_t t0;  // canonical index of slot 0
};
struct OvsKeys {
  int n;
  short p1[3 * ADJ_MAX_BATCH], p2[3 * ADJ_MAX_BATCH], first[3 * ADJ_MAX_BATCH + 1];
  signed char slot[3 * ADJ_MAX_BATCH], mode[3 * ADJ_MAX_BATCH];  // contributions, key by key
};

// dOVS[P1][x][P2][y] += the contributions of its key, in order
__global__ void __launch_bounds__(256) k_y_ovs(const __grid_constant__ YParts Yp, const __grid_constant__ OvsKeys K,
                                               int o, int v, double* __restrict__ dOVS) {
  const int64_t e = blockIdx.x * 256LL + threadIdx.x, v2 = (int64_t)v * v;
  if (e >= v2) return;
  const int key = blockIdx.y, x = (int)(e / v), y = (int)(e - (int64_t)x * v);
  double s = 0.0;
  for (int c = K.first[key]; c < K.first[key + 1]; ++c) s += Yp.s[K.mode[c]][K.slot[c] * Yp.stride + e];
  dOVS[(((int64_t)K.p1[key] * v + x) * o + K.p2[key]) * v + y] += s;
}

__device__ double block_sum(const double* __restrict__ x, int n, double* red) {
  double s = 0.0;
  for (int e = threadIdx.x; e < n; e += 256) s += x[e];
  for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  double t = 0.0;
  for (int w = 0; w < 8; ++w) t += red[w];
  __syncthreads();
  return t;
}

// dt1, d eps and the shares of a batch, slot after slot
__global__ void __launch_bounds__(256) k_y_small(const __grid_constant__ AdjEpi A, const __grid_constant__ AdjBatch B,
                                                 const __grid_constant__ YParts Yp, const __grid_constant__ AdjOut O,
                                                 int agrid) {
  __shared__ double red[8];
  const int v = A.a.v;
  if (blockIdx.x == 0) {
    for (int s = 0; s < B.n; ++s) {
      const Triple T = B.t[s];
      const double e = block_sum(A.epart + (int64_t)s * agrid, agrid, red);
      const double d = block_sum(A.dpart + (int64_t)s * agrid, agrid, red);
      if (threadIdx.x == 0) {
        O.shares[O.t0 + s] = e * ((double)T.m / 3.0);
        if (O.eps_o) {
          O.eps_o[T.i] += d;
          O.eps_o[T.j] += d;
          O.eps_o[T.k] += d;
        }
      }
    }
    return;
  }
  const int z = (blockIdx.x - 1) * 256 + threadIdx.x;
  if (z >= v) return;
  for (int s = 0; s < B.n; ++s) {
    const Triple T = B.t[s];
    const int64_t so = s * Yp.stride;
    if (O.t1) {
      O.t1[(int64_t)T.k * v + z] += Yp.p[0][so + z];
      O.t1[(int64_t)T.i * v + z] += Yp.q[0][so + z];
      O.t1[(int64_t)T.j * v + z] += Yp.p[1][so + z];
    }
    if (O.eps_v) O.eps_v[z] -= Yp.q[1][so + z] + (Yp.p[2][so + z] + Yp.p[3][so + z]);
  }
}

// ---------------------------------------------------------------------------
// slices of dW~
// ---------------------------------------------------------------------------

// Slices of index permutations of dW~ into layouts L[x][y][z] (z padded to vp),
// permutation q holding the slices of dW~[pi_q(x, y, z)]:
//   0, 1, 2: pi = (x,y,z), (z,x,y), (y,z,x);  3, 4, 5: (z,y,x), (x,z,y), (y,x,z).
// With 2^e > max |dW~| (e written to e_out) the digits are slice_digits_int's (integer
// operations on the bits of dW~).  A block takes a 16 x 16 x 16 cube of dW~: each
// value is read and cut once, and every layout is written from shared memory in
// rows of 16 elements (32 bytes); 64 consecutive blocks take a cube of 64^3, so that
// the pieces of a 128-byte line meet in L2 in every layout.  HBM bounds it: 8 bytes
// read and 2 NS written per value and layout; one triple at nvir = 320: 0.55 ms (0.82 with
// the blocks in row order, whose pieces of the transposed layouts lie 400 blocks apart).
template <int NS>
__global__ void __launch_bounds__(256) k_dw_slices(const double* __restrict__ dWs, int64_t w_stride, int v, int vp,
                                                   int perm0, const unsigned long long* __restrict__ dwmax,
                                                   int* __restrict__ e_out, bf* __restrict__ out, int64_t lay_elems,
                                                   int64_t slot_elems, int nperm) {
  // [slice][i][j][k], rows of 16 elements on 18 and planes of 16 rows on 290: the
  // transposed reads below then spread over the banks
  constexpr int RS = 18, PS = 16 * RS + 2;
  __shared__ unsigned short cube[NS][16 * PS];
  const int slot = blockIdx.z;
  const double* dW = dWs + slot * w_stride;
  const double mx = __longlong_as_double((long long)dwmax[slot]);
  int ex = 0;
  if (mx > 0.0) frexp(mx, &ex);
  if (blockIdx.x == 0 && threadIdx.x == 0) e_out[slot] = ex;
  const int n4 = (v + 63) / 64, sub = blockIdx.x & 63, sup = blockIdx.x >> 6;
  const int a0 = sup / (n4 * n4) * 64 + (sub >> 4) * 16, b0 = sup / n4 % n4 * 64 + (sub >> 2 & 3) * 16,
            c0 = sup % n4 * 64 + (sub & 3) * 16;
  if (a0 >= v || b0 >= v || c0 >= v) return;
  const int64_t V = v, plane = V * V * vp;
  const int k = threadIdx.x & 15, j0 = threadIdx.x >> 4;
#pragma unroll 4
  for (int i = 0; i < 16; ++i) {
    const bool in = a0 + i < v && b0 + j0 < v && c0 + k < v;
    int d[NS];
    slice_digits_int<NS>(in ? dW[((int64_t)(a0 + i) * V + b0 + j0) * V + c0 + k] : 0.0, ex, d);
#pragma unroll
    for (int s = 0; s < NS; ++s) cube[s][i * PS + j0 * RS + k] = (unsigned short)digit_bf16(d[s], 7 * (s + 1));
  }
  __syncthreads();
  // Output rows: (x, y) fixed, z along the row; thread = (row, half of 8 elements).
  // In terms of the cube's (i, j, k) = offsets of dW~'s (first, second, third) index
  const int half = threadIdx.x & 1, r0 = threadIdx.x >> 1;
  for (int q = 0; q < nperm; ++q) {
    const int perm = perm0 + q;
    // which of dW~'s indices (0, 1, 2) are x, y and z
    const int px = perm == 0 ? 0 : perm == 1 ? 1 : perm == 2 ? 2 : perm == 3 ? 2 : perm == 4 ? 0 : 1;
    const int py = perm == 0 ? 1 : perm == 1 ? 2 : perm == 2 ? 0 : perm == 3 ? 1 : perm == 4 ? 2 : 0;
    const int pz = 3 - px - py;
    auto org = [&](int p) { return p == 0 ? a0 : (p == 1 ? b0 : c0); };
    auto stp = [&](int p) { return p == 0 ? PS : (p == 1 ? RS : 1); };
    const int x0 = org(px), y0 = org(py), z0 = org(pz), sx = stp(px), sy = stp(py), sz = stp(pz);
    bf* o = out + slot * slot_elems + q * lay_elems;
#pragma unroll
    for (int rr = 0; rr < 2; ++rr) {
      const int r = r0 + 128 * rr, x = r >> 4, y = r & 15, zz = 8 * half;
      if (x0 + x >= v || y0 + y >= v || z0 + zz >= vp) continue;
      const int at = x * sx + y * sy + zz * sz;
      bf* dst = o + ((int64_t)(x0 + x) * V + y0 + y) * vp + z0 + zz;  // vp and z0 + zz are multiples of 8
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        uint32_t w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          w[u] = (uint32_t)cube[s][at + 2 * u * sz] | ((uint32_t)cube[s][at + (2 * u + 1) * sz] << 16);
        *reinterpret_cast<uint4*>(dst + s * plane) = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
  }
}

int64_t rup(int64_t x, int64_t m) { return (x + m - 1) / m * m; }

// Slices per element: four (28 bits) up to nvir = 200, five (35 bits) above.
// The back-contractions sum v (or v^2) products whose largest terms can sit far
// above the result, and the rows of t2 and ovvv away from the occupied-virtual
// boundary far below their scale; at nocc=48 nvir=560 four slices left errors
// of 2.7e-6 of d ovvv's largest entry.
int adjoint_slices(int64_t v) { return v > 200 ? 5 : 4; }

struct AdjPlan {
  bool full;
  int B, ns, vp;
  size_t lay;      // elements of one dW~ layout (ns planes of v v vp)
  size_t region;   // bytes per slot: G, dY and dD, later the layouts
  size_t ovt, t2t, t2p, noo;  // bytes of the operand transposes
  int64_t ystride;  // doubles of YParts per slot
  int64_t part_cap; // doubles of split-K partials
  size_t bytes;
};

size_t al(size_t b) { return (b + 1023) & ~size_t(1023); }

AdjPlan adj_plan(int64_t o, int64_t v, int num_sms, bool full) {
  AdjPlan z;
  z.full = full;
  z.ns = adjoint_slices(v);
  z.vp = (int)rup(v, 16);
  const int64_t v3 = v * v * v, vp = z.vp, NS = z.ns, nt = num_unique_triples(o);
  z.lay = (size_t)NS * v * v * vp;
  const int nlay = full ? 6 : 3;
  z.region = std::max(al((size_t)3 * v3 * 8) + 2 * al((size_t)v3 * 8), (size_t)nlay * al(z.lay * 2));
  z.B = 1;
  if (full) {
    const int64_t per = (int64_t)z.region + 8 * v3;
    z.B = (int)std::max<int64_t>(1, std::min<int64_t>({ADJ_MAX_BATCH, ADJ_BATCH_BYTES / per, std::max<int64_t>(1, nt)}));
  }
  const int64_t npair = full ? o * o : 6, nocc = full ? o : 3, nslab = full ? o : 1;
  z.ovt = al((size_t)nslab * NS * v * v * vp * 2);
  z.t2t = al((size_t)npair * NS * v * vp * 2);
  z.t2p = al((size_t)nocc * NS * o * v * vp * 2);
  z.noo = al((size_t)NS * o * o * o * vp * 2);
  z.ystride = rup(7 * v * v + 2 * v, 4);
  // partials of the split jobs of one launch: an upper bound over the launches, or
  // in the lean form (one slab and three ooov blocks per launch) about that, less
  // what the Y parts take; vt_finish fits its split counts to it
  const int64_t ntv = vt_ntile(v, false), nto = vt_ntile(o, false), rows_z = (v + 127) / 128;
  const int64_t pair_blk = (full ? 6 * z.B : 3) * vt_seg_blocks((int)v, (int)v, VT_SPLIT_CHUNKS);
  const int64_t d_ooov = vt_split_doubles(rows_z * ((o + nto - 1) / nto), pair_blk, v * o, num_sms);
  const int64_t d_t2 = vt_split_doubles(rows_z * ((v + ntv - 1) / ntv), pair_blk, v * v, num_sms);
  if (full) z.part_cap = 6 * (d_t2 + d_ooov + 16) + 1024;
  else z.part_cap = std::max<int64_t>(64, 3 * (d_t2 + d_ooov) + 1024 - z.ystride);
  z.bytes = tc_slices_bytes((int)o, (int)v, z.ns) + 1024 + 2 * al((size_t)o * v * o * v * 8) /* ovs, dOVS */ +
            z.B * (al(z.region) + al((size_t)v3 * 8)) + 2 * al((size_t)z.B * adjoint_grid(num_sms) * 8) +
            al((size_t)std::max<int64_t>(1, nt) * 8) + al(256) + al((size_t)z.B * z.ystride * 8) + z.ovt + z.t2t + z.t2p + z.noo +
            al((size_t)z.part_cap * 8) + 4096;
  return z;
}

// The forms of a gradient, best first.  All transposes at hand where they (and six
// layouts for three) take at most ADJ_FULL_BYTES more: per triple of nocc=32
// nvir=320 7.6 ms against 9.7 in the lean form (13.3 before there were two).
std::vector<AdjPlan> adj_forms(const Handle* h, int64_t o, int64_t v) {
  const AdjPlan lean = adj_plan(o, v, h->num_sms, false), full = adj_plan(o, v, h->num_sms, true);
  const int64_t more = (int64_t)(full.bytes - lean.bytes) - 8 * (full.part_cap - lean.part_cap);
  if (more > ADJ_FULL_BYTES) return {lean};
  return {full, lean};
}

std::vector<size_t> plan_bytes(const std::vector<AdjPlan>& f) {
  std::vector<size_t> b;
  for (const AdjPlan& z : f) b.push_back(z.bytes);
  return b;
}

}  // namespace

std::vector<size_t> vjp_tc_bytes(const Handle* h, int64_t o, int64_t v) { return plan_bytes(adj_forms(h, o, v)); }

// The contractions of one triple (g = 0, 1, 2 the G blocks with occupied
// indices (p, q, r) = (i, j, k), (j, k, i), (k, i, j); dG_g the views of dW~):
//   G:  G_g[x,y,z] = S1 + S2 + S3 + S4 (four K segments, the forward's form)
//   (a) dovvv[p,x,y,d] += sum_z dG[x,y,z] t2[r,q,z,d]    (b) dovvv[q,y,x,d] += sum_z dG[x,y,z] t2[r,p,z,d]
//   (c) dt2[r,q,z,d] += sum_xy dG[x,y,z] ovvv[p,x,y,d]   (d) dt2[r,p,z,d] += sum_xy dG[x,y,z] ovvv[q,y,x,d]
//   (e) dt2[l,p,y,x] -= sum_z dG[x,y,z] ooov[q,l,r,z]    (g) dt2[l,q,x,y] -= sum_z dG[x,y,z] ooov[p,l,r,z]
//   (f) dooov[q,l,r,z] -= sum_xy t2[l,p,y,x] dG[x,y,z]   (h) dooov[p,l,r,z] -= sum_xy t2[l,q,x,y] dG[x,y,z]
// Every operand is read along a contiguous K index: dG_g comes in the layouts
// L1_g[x][y][z] (K = z), L2_g[z][x][y] (K = (x, y)) and L3_g[z][y][x] (K =
// (y, x)), the index permutations of dW~ that k_dw_slices writes; t2, ovvv
// and ooov enter as transposed slice copies (t2T[d][z] per pair (r, q),
// ovvvT[d][x][y] per slab, t2P[l][x][y] per occupied index, nooTT[q][r][l][z]).
// G and (a), (b), (e), (g) run on pairs of CTAs; (c), (d), (f), (h) have one row
// tile (z) and run on lone CTAs, split over K.  Outputs of the same launch are
// disjoint: the contributions to one output slab (or pair block) are the
// segments of one job.
te_status run_vjp_tc(Handle* h, const te_cluster* c, int64_t t_begin, int64_t t_end, double gE,
                     double* e_out, te_cluster_grad* g, cudaStream_t s, int64_t cluster) {
  const int o = (int)c->nocc, v = (int)c->nvir;
  const int64_t v2 = (int64_t)v * v, v3 = v2 * v, nt = num_unique_triples(o);
  const std::vector<AdjPlan> forms = adj_forms(h, o, v);
  size_t form = 0;
  te_status st = acquire_workspace(h, plan_bytes(forms), &form);
  if (st != TE_OK) return st;
  const AdjPlan Z = forms[form];
  st = ensure_triples_public(h, o);
  if (st != TE_OK) return st;
  const int ns = Z.ns;
  const int64_t vp = Z.vp, O = o, V = v, NS = ns;
  char* base = reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(h->ws) + 1023) & ~uintptr_t(1023));
  char* p = base + al(tc_slices_bytes(o, v, ns));
  auto takeb = [&](size_t bytes) {
    char* r = p;
    p += al(bytes);
    return r;
  };
  auto take = [&](int64_t n) { return reinterpret_cast<double*>(takeb((size_t)n * 8)); };
  double* ovs = take((int64_t)o * v * o * v);
  char* region = takeb(Z.B * al(Z.region));
  double* dW = reinterpret_cast<double*>(takeb(Z.B * al((size_t)v3 * 8)));
  double* dOVS = take((int64_t)o * v * o * v);
  const int agrid = adjoint_grid(h->num_sms);
  double* epart = take((int64_t)Z.B * agrid);
  double* dpart = take((int64_t)Z.B * agrid);
  double* shares = take(std::max<int64_t>(1, nt));
  unsigned long long* dwmax = reinterpret_cast<unsigned long long*>(takeb(256));
  int* dwexp = reinterpret_cast<int*>(dwmax + ADJ_MAX_BATCH);
  double* ypart = take(Z.B * Z.ystride);
  bf* ovT = reinterpret_cast<bf*>(takeb(Z.ovt));
  bf* t2T = reinterpret_cast<bf*>(takeb(Z.t2t));
  bf* t2P = reinterpret_cast<bf*>(takeb(Z.t2p));
  bf* nooTT = reinterpret_cast<bf*>(takeb(Z.noo));
  double* part = take(Z.part_cap);
  const int64_t reg_stride = (int64_t)al(Z.region);                // bytes per slot
  const int64_t lay_stride = (int64_t)al(Z.lay * 2) / 2;           // elements between layouts of a slot

  SliceSet S;
  st = tc_prepare_slices(c, base, &S, h->num_sms, s, ns, h->d_err, cluster, &h->n_launches);
  if (st != TE_OK) return st;
  Prepared P{};  // float64 ovs for the disconnected term
  P.ovs = ovs;
  cudaError_t e = launch_prep_fp64(c, &P, s);
  ++h->n_launches;

  auto zero = [&](double* ptr, int64_t n) {
    if (ptr && e == cudaSuccess) e = cudaMemsetAsync(ptr, 0, sizeof(double) * n, s);
  };
  zero(g->eps_o, o);
  zero(g->eps_v, v);
  zero(g->ovvv, (int64_t)o * v3);
  zero(g->ooov, (int64_t)o * o * o * v);
  zero(g->ovov, (int64_t)o * v * o * v);
  zero(g->t1, (int64_t)o * v);
  zero(g->t2, (int64_t)o * o * v2);
  zero(dOVS, (int64_t)o * v * o * v);
  if (e != cudaSuccess) return fail(TE_ECUDA, "gradient setup: %s", cudaGetErrorString(e));

  const bf* sO = static_cast<const bf*>(S.ovvv);
  const bf* sT = static_cast<const bf*>(S.t2);
  const bf* sL = static_cast<const bf*>(S.t2L);
  const bf* sN = static_cast<const bf*>(S.nooT);
  const int64_t op = S.op;
  // nooTT[q][r][l][z] = nooT[q][r][z][l] = -ooov[q,l,r,z], once per call
  auto transpose_t2P = [&](int q, bf* dst) {
    ++h->n_launches;
    return vt_transpose(sL + (int64_t)q * S.t2L_q, S.t2L_plane, V * op, op, dst, O * V * vp, vp, V * vp, ns, v, v, o, s);
  };
  auto transpose_slab = [&](int sb, bf* dst) {
    ++h->n_launches;
    return vt_transpose(sO + (int64_t)sb * S.ovvv_p, S.ovvv_plane, V * vp, vp, dst, V * V * vp, vp, V * vp, ns, v, v, v, s);
  };
  e = vt_transpose(sN, S.nooT_plane, S.nooT_pr, op, nooTT, O * O * O * vp, O * vp, vp, ns, o * o, v, o, s);
  ++h->n_launches;
  if (Z.full && t_end > t_begin) {
    if (e == cudaSuccess) e = vt_transpose(sT, S.t2_plane, S.t2_rq, vp, t2T, V * vp, NS * V * vp, vp, ns, o * o, v, v, s);
    ++h->n_launches;
    for (int q = 0; q < o && e == cudaSuccess; ++q) e = transpose_t2P(q, t2P + q * NS * O * V * vp);
    for (int q = 0; q < o && e == cudaSuccess; ++q) e = transpose_slab(q, ovT + q * NS * V * V * vp);
  }
  if (e != cudaSuccess) return fail(TE_ECUDA, "transpose: %s", cudaGetErrorString(e));

  // tensor maps, encoded once: rows (x, y) in tiles of 8 x 16, rows z alone in
  // tiles of 128; B rows by halves of a tile for the pair launches
  const int NTv = vt_ntile(v, false), NTo = vt_ntile(o, false);  // lone launches
  const int NPv = vt_ntile(v, true), NPo = vt_ntile(o, true);  // pair launches
  VtBank bank;
  bank.n = 0;
  auto add = [&](const void* b0, std::initializer_list<int64_t> dims, std::initializer_list<int64_t> str,
                 VtRoles r, int rows2, int rows1, int* idx) {
    VtView w;
    w.base = b0;
    int q = 0;
    for (int64_t d : dims) w.dims[q++] = (uint64_t)d;
    q = 0;
    for (int64_t x : str) w.stride[q++] = (uint64_t)x;
    w.roles = r;
    return vt_bank_add(&bank, w, rows2, rows1, idx);
  };
  const VtRoles XY{0, 1, 2, -1, 3, 0};       // k2 | rows y, x | slice | group
  const VtRoles ROW{0, 1, -1, -1, 2, 0};     // k2 | rows | slice | groups
  const VtRoles ZK{0, 2, -1, 1, 3, 0};       // k2 | k1 | rows | slice | group
  int m_g[6], m_l1n[3], m_l1t[3], m_l2[3], m_l3[3], m_t2T, m_noo, m_ovT, m_t2P;
  const int64_t U1 = 1, NB = Z.B, ls = reg_stride / 2;  // elements between the slots' layouts
  if ((st = vt_slice_maps(&bank, S, o, v, NPv, m_g)) != TE_OK) return st;
  const int m_on = m_g[0], m_ot = m_g[1], m_ln = m_g[2], m_lt = m_g[3], m_t2 = m_g[4], m_no = m_g[5];
  const int64_t lplane = V * V * vp;
  // L1_g and L2_g are permutations 0..2 (L2_g is the one of G block (g + 2) % 3), L3_g permutations 3..5
  const bf* lay = reinterpret_cast<bf*>(region);
  const int l2perm[3] = {2, 0, 1};
  auto lay_of = [&](int perm) { return lay + (Z.full ? perm : perm % 3) * lay_stride; };
  for (int q = 0; q < 3; ++q) {
    if ((st = add(lay_of(q), {V, V, V, NS, NB}, {1, vp, V * vp, lplane, ls}, XY, 16, 8, &m_l1n[q])) != TE_OK) return st;
    if ((st = add(lay_of(q), {V, V, V, NS, NB}, {1, V * vp, vp, lplane, ls}, XY, 16, 8, &m_l1t[q])) != TE_OK) return st;
    if ((st = add(lay_of(l2perm[q]), {V, V, V, NS, NB}, {1, vp, V * vp, lplane, ls}, ZK, 128, 1, &m_l2[q])) != TE_OK)
      return st;
    if ((st = add(lay_of(3 + q), {V, V, V, NS, NB}, {1, vp, V * vp, lplane, ls}, ZK, 128, 1, &m_l3[q])) != TE_OK)
      return st;
  }
  const int64_t npx = Z.full ? O : 6, npy = Z.full ? O : 1;  // t2T[r][q] or slots
  if ((st = add(t2T, {V, V, NS, npx, npy}, {1, vp, V * vp, NS * V * vp, npx * NS * V * vp}, ROW, NPv / 2, 1, &m_t2T)) != TE_OK)
    return st;
  if ((st = add(nooTT, {V, O, O, O, NS}, {1, vp, O * vp, O * O * vp, O * O * O * vp}, VtRoles{0, 1, -1, -1, 4, 0}, NPo / 2,
                1, &m_noo)) != TE_OK)
    return st;
  if ((st = add(ovT, {V, V, V, NS, Z.full ? O : U1}, {1, vp, V * vp, V * V * vp, NS * V * V * vp}, ZK, NTv, 1, &m_ovT)) !=
      TE_OK)
    return st;
  if ((st = add(t2P, {V, V, O, NS, Z.full ? O : 3 * U1}, {1, vp, V * vp, O * V * vp, NS * O * V * vp}, ZK, NTo, 1,
                &m_t2P)) != TE_OK)
    return st;

  auto eO = [&](int p_) { return S.e_ovvv + p_; };
  auto eT = [&](int r_, int q_) { return S.e_t2 + ((int64_t)r_ * o + q_); };
  auto eL = [&](int q_) { return S.e_t2L + q_; };
  auto eN = [&](int p_, int r_) { return S.e_nooT + ((int64_t)p_ * o + r_); };

  AdjEpi A;
  A.a = AdjArgs{};
  A.a.o = o;
  A.a.v = v;
  A.a.G = reinterpret_cast<const double*>(region);
  A.a.ovs = ovs;
  A.a.t1 = c->t1;
  A.a.eps_o = c->eps_o;
  A.a.eps_v = c->eps_v;
  A.dY = reinterpret_cast<double*>(region + al((size_t)3 * v3 * 8));
  A.dD = A.dY + al((size_t)v3 * 8) / 8;
  A.dW = dW;
  A.g_stride = A.d_stride = reg_stride / 8;
  A.w_stride = (int64_t)al((size_t)v3 * 8) / 8;
  A.dwmax = dwmax;
  A.epart = epart;
  A.dpart = dpart;
  YParts Yp;
  for (int q = 0; q < 3; ++q) Yp.s[q] = ypart + q * v2;
  for (int q = 0; q < 4; ++q) Yp.p[q] = ypart + (3 + q) * v2;
  for (int q = 0; q < 2; ++q) Yp.q[q] = ypart + 7 * v2 + q * V;
  Yp.stride = Z.ystride;

  std::vector<Triple> trip = unique_triples(o);
  VtBuild* bp = new (std::nothrow) VtBuild;
  if (!bp) return fail(TE_ENOMEM, "view GEMM tables");
  VtBuild& b = *bp;
  struct Del {
    VtBuild* b;
    ~Del() { delete b; }
  } del{bp};
  auto launch = [&]() -> te_status {
    if (b.P.njobs == 0) return TE_OK;
    te_status q = vt_finish(&b, h->num_sms, part, Z.part_cap, nullptr);
    return q != TE_OK ? q : vt_launch(h, &b, s);
  };
  int slab = -1;  // lean: the ovvv slab whose transpose ovT holds
  auto need_slab = [&](int sb) -> cudaError_t {
    if (Z.full || slab == sb) return cudaSuccess;
    slab = sb;
    return transpose_slab(sb, ovT);
  };
  // one K segment of a lone-CTA job, grouped by its output block
  struct Piece {
    int amap, slot, bmap, bidx;
    const int* eb;
    int sign;
  };
  using Pieces = std::map<int, std::vector<Piece>>;
  for (int64_t t0 = t_begin; t0 < t_end && e == cudaSuccess; t0 += Z.B) {
    AdjBatch Bt{};
    Bt.n = (int)std::min<int64_t>(Z.B, t_end - t0);
    int PQR[ADJ_MAX_BATCH][3][3];
    for (int x = 0; x < Bt.n; ++x) {
      const Triple T = Bt.t[x] = trip[t0 + x];
      const int q[3][3] = {{T.i, T.j, T.k}, {T.j, T.k, T.i}, {T.k, T.i, T.j}};
      for (int gi = 0; gi < 3; ++gi)
        for (int d = 0; d < 3; ++d) PQR[x][gi][d] = q[gi][d];
      Bt.w[x] = gE * (double)T.m / 3.0;
    }
    // lean: slots of the transposes this triple reads
    int pr_[6][2], npair = 0, occ[3], nocc_ = 0;
    auto pair_slot = [&](int r_, int q_) {
      for (int x = 0; x < npair; ++x)
        if (pr_[x][0] == r_ && pr_[x][1] == q_) return x;
      pr_[npair][0] = r_;
      pr_[npair][1] = q_;
      return npair++;
    };
    auto occ_slot = [&](int x_) {
      if (Z.full) return x_;
      for (int q = 0; q < nocc_; ++q)
        if (occ[q] == x_) return q;
      occ[nocc_] = x_;
      return nocc_++;
    };
    if (!Z.full) {
      for (int gi = 0; gi < 3; ++gi) {
        pair_slot(PQR[0][gi][2], PQR[0][gi][1]);
        pair_slot(PQR[0][gi][2], PQR[0][gi][0]);
        occ_slot(PQR[0][gi][0]);
      }
      for (int x = 0; x < npair && e == cudaSuccess; ++x) {
        e = vt_transpose(sT + ((int64_t)pr_[x][0] * o + pr_[x][1]) * S.t2_rq, S.t2_plane, 0, vp, t2T + x * NS * V * vp,
                         V * vp, 0, vp, ns, 1, v, v, s);
        ++h->n_launches;
      }
      for (int x = 0; x < nocc_ && e == cudaSuccess; ++x) e = transpose_t2P(occ[x], t2P + x * NS * O * V * vp);
      if (e != cudaSuccess) break;
    }

    // forward G blocks, float64 [slot][g][x][y][z]
    vt_begin(&b, ns, true);
    for (int x = 0; x < Bt.n; ++x)
      for (int gi = 0; gi < 3; ++gi) {
        const int pp = PQR[x][gi][0], qq = PQR[x][gi][1], rr = PQR[x][gi][2];
        vt_job(&b, v, v, v, 8, 16, NPv, reinterpret_cast<double*>(region) + x * A.g_stride + gi * v3, v2, v, 1, VT_STORE);
        const int f_p[3] = {0, 0, pp}, f_q[3] = {0, 0, qq};
        const int t_qr[3] = {0, qq, rr}, t_pr[3] = {0, pp, rr}, n_rq[3] = {0, rr, qq}, n_rp[3] = {0, rr, pp};
        vt_seg(&b, vt_use(&b, bank, m_on), vt_use(&b, bank, m_t2), 1, v, f_p, t_qr, eO(pp), eT(rr, qq), 1);
        vt_seg(&b, vt_use(&b, bank, m_ot), vt_use(&b, bank, m_t2), 1, v, f_q, t_pr, eO(qq), eT(rr, pp), 1);
        vt_seg(&b, vt_use(&b, bank, m_lt), vt_use(&b, bank, m_no), 1, o, f_p, n_rq, eL(pp), eN(qq, rr), 1);
        vt_seg(&b, vt_use(&b, bank, m_ln), vt_use(&b, bank, m_no), 1, o, f_q, n_rp, eL(qq), eN(pp, rr), 1);
      }
    if ((st = launch()) != TE_OK) return st;
    e = cudaMemsetAsync(dwmax, 0, 8 * (size_t)Z.B, s);
    if (e != cudaSuccess) break;
    k_adjoint_batch<<<dim3((unsigned)agrid, (unsigned)Bt.n), 256, 0, s>>>(A, Bt);
    // the Y and denominator parts; G, dY and dD are dead afterwards and their
    // memory takes the dW~ layouts
    k_y_planes<<<dim3((unsigned)v, (unsigned)Bt.n), 256, 0, s>>>(A, Bt, Yp);
    k_y_columns<<<dim3((unsigned)((v + 31) / 32), (unsigned)Bt.n, 4), 256, 0, s>>>(Yp, v);
    h->n_launches += 3;
    if (g->ovov) {
      k_y_sum_a<<<dim3((unsigned)((v2 + 255) / 256), (unsigned)Bt.n), 256, 0, s>>>(A, Bt, Yp);
      OvsKeys K{};
      std::map<int, std::vector<std::pair<int, int>>> keys;  // (P1, P2) -> (slot, mode) in order
      for (int x = 0; x < Bt.n; ++x) {
        const Triple T = Bt.t[x];
        keys[T.i * o + T.j].emplace_back(x, 0);
        keys[T.j * o + T.k].emplace_back(x, 1);
        keys[T.i * o + T.k].emplace_back(x, 2);
      }
      int cn = 0;
      for (const auto& kv : keys) {
        K.p1[K.n] = (short)(kv.first / o);
        K.p2[K.n] = (short)(kv.first % o);
        K.first[K.n++] = (short)cn;
        for (const auto& sm : kv.second) {
          K.slot[cn] = (signed char)sm.first;
          K.mode[cn++] = (signed char)sm.second;
        }
      }
      K.first[K.n] = (short)cn;
      k_y_ovs<<<dim3((unsigned)((v2 + 255) / 256), (unsigned)K.n), 256, 0, s>>>(Yp, K, o, v, dOVS);
      h->n_launches += 2;
    }
    k_y_small<<<1 + (v + 255) / 256, 256, 0, s>>>(A, Bt, Yp, AdjOut{g->eps_o, g->eps_v, g->t1, dOVS, shares, t0}, agrid);
    ++h->n_launches;
    auto slices = [&](int perm0, int nperm) {
      const unsigned n4 = (unsigned)((v + 63) / 64);
      const dim3 grid(64 * n4 * n4 * n4, 1, (unsigned)Bt.n);
      bf* out = reinterpret_cast<bf*>(region);
      if (ns == 5)
        k_dw_slices<5><<<grid, 256, 0, s>>>(dW, A.w_stride, v, (int)vp, perm0, dwmax, dwexp, out, lay_stride, ls, nperm);
      else
        k_dw_slices<4><<<grid, 256, 0, s>>>(dW, A.w_stride, v, (int)vp, perm0, dwmax, dwexp, out, lay_stride, ls, nperm);
      ++h->n_launches;
    };
    slices(0, Z.full ? 6 : 3);
    if ((e = cudaGetLastError()) != cudaSuccess) break;

    // d ovvv (a, b) and d t2 slabs from ooov (e, g): layouts L1
    vt_begin(&b, ns, true);
    std::vector<int> dist;
    for (int x = 0; x < Bt.n; ++x)
      for (int y : {Bt.t[x].i, Bt.t[x].j, Bt.t[x].k})
        if (std::find(dist.begin(), dist.end(), y) == dist.end()) dist.push_back(y);
    for (int sb : dist) {
      if (!g->ovvv) break;
      vt_job(&b, v, v, v, 8, 16, NPv, g->ovvv + (int64_t)sb * v3, v2, v, 1, VT_ADD);
      for (int x = 0; x < Bt.n; ++x)
        for (int gi = 0; gi < 3; ++gi) {
          const int pp = PQR[x][gi][0], qq = PQR[x][gi][1], rr = PQR[x][gi][2];
          const int fs[3] = {0, 0, x};
          const int f_rq[3] = {0, Z.full ? qq : (pp == sb ? pair_slot(rr, qq) : 0), Z.full ? rr : 0};
          const int f_rp[3] = {0, Z.full ? pp : (qq == sb ? pair_slot(rr, pp) : 0), Z.full ? rr : 0};
          if (pp == sb) vt_seg(&b, vt_use(&b, bank, m_l1n[gi]), vt_use(&b, bank, m_t2T), 1, v, fs, f_rq, dwexp + x, eT(rr, qq), 1);
          if (qq == sb) vt_seg(&b, vt_use(&b, bank, m_l1t[gi]), vt_use(&b, bank, m_t2T), 1, v, fs, f_rp, dwexp + x, eT(rr, pp), 1);
        }
    }
    for (int sb : dist) {
      if (!g->t2) break;
      // element dt2[l][sb][X][Y]: rows (X, Y), columns l
      vt_job(&b, v, v, o, 8, 16, NPo, g->t2 + (int64_t)sb * v2, v, 1, (int64_t)o * v2, VT_ADD);
      for (int x = 0; x < Bt.n; ++x)
        for (int gi = 0; gi < 3; ++gi) {
          const int pp = PQR[x][gi][0], qq = PQR[x][gi][1], rr = PQR[x][gi][2];
          const int fs[3] = {0, 0, x}, f_rq[3] = {rr, qq, 0}, f_rp[3] = {rr, pp, 0};
          // (e): X = y, Y = x: transposed rows; B = nooTT = -ooov
          if (pp == sb) vt_seg(&b, vt_use(&b, bank, m_l1t[gi]), vt_use(&b, bank, m_noo), 1, v, fs, f_rq, dwexp + x, eN(qq, rr), 1);
          if (qq == sb) vt_seg(&b, vt_use(&b, bank, m_l1n[gi]), vt_use(&b, bank, m_noo), 1, v, fs, f_rp, dwexp + x, eN(pp, rr), 1);
        }
    }
    if ((st = launch()) != TE_OK) return st;

    // d t2 pair blocks from ovvv (c), (d) and d ooov (h), (f): layouts L2, L3
    auto t2_piece = [&](Pieces& P, int x, int gi, bool d) {
      const int pp = PQR[x][gi][0], qq = PQR[x][gi][1], rr = PQR[x][gi][2], sb = d ? qq : pp;
      P[rr * o + (d ? pp : qq)].push_back(Piece{d ? m_l3[gi] : m_l2[gi], x, m_ovT, Z.full ? sb : 0, eO(sb), 1});
    };
    auto ooov_piece = [&](Pieces& P, int x, int gi, bool f) {
      const int pp = PQR[x][gi][0], qq = PQR[x][gi][1], rr = PQR[x][gi][2], src = f ? pp : qq;
      P[(f ? qq : pp) * o + rr].push_back(Piece{f ? m_l3[gi] : m_l2[gi], x, m_t2P, occ_slot(src), eL(src), -1});
    };
    auto jobs = [&](const Pieces& P, bool t2out) {
      for (const auto& kv : P) {
        const int r_ = kv.first / o, q_ = kv.first % o;
        if (t2out) vt_job(&b, 1, v, v, 1, 128, NTv, g->t2 + ((int64_t)r_ * o + q_) * v2, 0, v, 1, VT_ADD);
        else vt_job(&b, 1, v, o, 1, 128, NTo, g->ooov + ((int64_t)r_ * o * o + q_) * v, 0, 1, (int64_t)o * v, VT_ADD);
        for (const Piece& w : kv.second) {
          const int fa[3] = {0, 0, w.slot}, fb[3] = {0, 0, w.bidx};
          vt_seg(&b, vt_use(&b, bank, w.amap), vt_use(&b, bank, w.bmap), v, v, fa, fb, dwexp + w.slot, w.eb, w.sign);
        }
      }
    };
    if (Z.full) {
      Pieces P2, Po;
      for (int x = 0; x < Bt.n; ++x)
        for (int gi = 0; gi < 3; ++gi)
          for (int k = 0; k < 2; ++k) {
            if (g->t2) t2_piece(P2, x, gi, k == 1);
            if (g->ooov) ooov_piece(Po, x, gi, k == 1);
          }
      vt_begin(&b, ns, false);
      jobs(P2, true);
      jobs(Po, false);
      if ((st = launch()) != TE_OK) return st;
      continue;
    }
    // lean: one slab transpose per launch; L2 with (c) and (h), then L3 with (d)
    // and (f), slabs in reverse order (the last slab of (c) is still transposed)
    const int order[3] = {PQR[0][0][0], PQR[0][0][1], PQR[0][0][2]};
    for (int k = 0; k < 2 && e == cudaSuccess; ++k) {
      if (k == 1) slices(3, 3);
      bool first = true;
      for (int q = 0; q < 3 && e == cudaSuccess; ++q) {
        const int at = k == 0 ? q : 2 - q, sb = order[at];
        bool seen = false;
        for (int y = 0; y < q; ++y) seen |= order[k == 0 ? y : 2 - y] == sb;
        if (seen) continue;
        Pieces P2, Po;
        for (int gi = 0; gi < 3; ++gi) {
          if (g->t2 && PQR[0][gi][k] == sb) t2_piece(P2, 0, gi, k == 1);
          if (g->ooov && first) ooov_piece(Po, 0, gi, k == 1);
        }
        first = false;
        vt_begin(&b, ns, false);
        jobs(P2, true);
        jobs(Po, false);
        if (!P2.empty() && (e = need_slab(sb)) != cudaSuccess) break;
        if ((st = launch()) != TE_OK) return st;
      }
    }
    if (e == cudaSuccess) e = cudaGetLastError();
  }
  if (e == cudaSuccess && g->ovov) {
    e = launch_dovov(o, v, dOVS, g->ovov, s);
    ++h->n_launches;
  }
  if (e == cudaSuccess && e_out) {
    e = launch_reduce_total(shares + t_begin, t_end - t_begin, e_out, s);
    ++h->n_launches;
  }
  if (e != cudaSuccess) return fail(TE_ECUDA, "vjp launch: %s", cudaGetErrorString(e));
  return TE_OK;
}

}  // namespace te
