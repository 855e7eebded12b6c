// Energy epilogue of the tensor-core modes: a persistent kernel fed by TMA.
//
// Work item = (triple slot, block triple X >= Y >= Z of 8-wide virtual
// blocks).  The contraction kernel stores G orbit-major (energy_tc.h): the
// item's 18 G cubes (3 G blocks x 6 block orders) are contiguous and arrive
// by one bulk copy; the 18 8x8 blocks of the symmetrised ovov the item uses
// and 9 t1 rows come by TMA (few, large copies: the copy engine's per-copy
// cost, not HBM, limited a layout that needed 54 copies per item).  A
// producer warp issues the loads into a double buffer; one thread per
// orbit candidate (a,b,c) of the 8^3 block triple.  G is either FP32 (BF16X3/TF32/TF32X3) or an FP32 pair
// hi + lo (OZAKI), CW = 1 or 2 floats per element.
//
// Orbit sum without cancellation: the 6x6 coefficient matrix C of R between
// the six orbit positions (T = sum_nm W_n C_nm V_m) has zero row and column
// sums, so T is unchanged when W_0 and V_0 are subtracted from every
// position.  The deviations w_n = W_n - W_0 are formed G block by G block
// (differences of close FP32 numbers are nearly exact), so the symmetric
// part of W~, which R annihilates, never enters a rounded product.
//   T = 3 sum_n w_n v_n + Ae Se + Ao So - 2 (Ae So + Ao Se)
// D, its reciprocal (FP32 seed + one Newton step in FP64: error ~1e-14),
// A T / D and the sums are FP64.
#include <cstring>

#include "energy_tc.h"
#include "ptx_sm100.cuh"

namespace te {

namespace {

constexpr int TB = 8;
constexpr int WARPS = 16;                 // compute warps: one orbit candidate (a,b,c) of 8^3 per thread
constexpr int THREADS = (WARPS + 1) * 32;  // + one producer warp

template <int CW>
struct Layout {
  static constexpr uint32_t cube_bytes = TB * TB * TB * 4 * CW;
  static constexpr uint32_t cubes = 18 * cube_bytes;
  static constexpr uint32_t ovs = 27 * TB * TB * 4;
  static constexpr uint32_t t1 = 9 * 128;
  static constexpr uint32_t eps = 640;  // dAB[64] = e_ijk - e_a - e_b, epsC[8] (FP64, written by the producer)
  static constexpr uint32_t buf = cubes + ovs + t1 + eps;
  static constexpr uint32_t tx = 18 * cube_bytes + 18 * TB * TB * 4 + 9 * TB * 4;
};

__device__ __forceinline__ void decode_bt(int64_t bt, int* blk) {
  // bt = X(X+1)(X+2)/6 + Y(Y+1)/2 + Z, X >= Y >= Z >= 0 (FP32 estimate, exact integer fix-up)
  int x = (int)cbrtf(6.0f * (float)bt);
  while (x > 0 && (int64_t)x * (x + 1) * (x + 2) / 6 > bt) --x;
  while ((int64_t)(x + 1) * (x + 2) * (x + 3) / 6 <= bt) ++x;
  const int64_t rem = bt - (int64_t)x * (x + 1) * (x + 2) / 6;
  int y = (int)sqrtf(2.0f * (float)rem);
  while (y > 0 && (int64_t)y * (y + 1) / 2 > rem) --y;
  while ((int64_t)(y + 1) * (y + 2) / 2 <= rem) ++y;
  blk[0] = x;
  blk[1] = y;
  blk[2] = (int)(rem - (int64_t)y * (y + 1) / 2);
}

// ---- double-float (pair of FP32) arithmetic: error-free transformations ----
// Knuth two-sum, FMA two-product; the rn intrinsics forbid contraction.
struct df {
  float h, l;
};

__device__ __forceinline__ df df_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}

__device__ __forceinline__ df df_norm(float h, float l) {
  const float s = __fadd_rn(h, l);
  return {s, __fsub_rn(l, __fsub_rn(s, h))};
}

__device__ __forceinline__ df df_add(df a, df b) {
  const df s = df_two_sum(a.h, b.h);
  return df_norm(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}

__device__ __forceinline__ df df_mul(df a, df b) {
  const float p = __fmul_rn(a.h, b.h);
  const float e = fmaf(a.h, b.h, -p);
  return df_norm(p, __fadd_rn(e, __fadd_rn(__fmul_rn(a.h, b.l), __fmul_rn(a.l, b.h))));
}

__device__ __forceinline__ df df_scale(df a, float k) {  // k a small integer
  const float p = __fmul_rn(a.h, k);
  const float e = fmaf(a.h, k, -p);
  return df_norm(p, __fadd_rn(e, __fmul_rn(a.l, k)));
}

struct EnergyMaps {
  CUtensorMap ovs[TC_MAX_CL];  // per cluster: ovs32 [o][v][o][vq], 4D (b, j, a, i)
  CUtensorMap t1[TC_MAX_CL];   // per cluster: t1 [o][vq], 2D (a, i)
};

struct EnergyParams {
  int ncl, npieces;
  int64_t items;
  EnergyCl cl[TC_MAX_CL];
  TcPiece pc[TC_MAX_PIECES];  // G: orbit-major [slot][bt][g][pid][CW planes][512, swizzled] from pc.gbuf
  const Triple* triples;
  double* partials;  // [slot][first item of the block][WARPS]: the warps' sums of a triple's items
  unsigned int* err;
  unsigned long long wait_ns;
};

struct PieceTable {
  int n;
  TcPiece pc[TC_MAX_PIECES];
};

// A block's items: item bt of canonical triple t belongs to block (t nbt + bt)
// mod gridDim.x, so consecutive triples follow each other around the blocks
// without a gap (restarting every triple at block 0 left 11% of the block
// slots empty at nvir = 120: 680 items on 152 blocks).  Which items of a
// triple a block takes, and in which order, depends on t, nbt and the grid
// size alone (the grid is always one block per SM), not on the launch's other
// pieces: a triple's float64 sums have the same bits in a single-cluster call
// and in a batch.
struct ItemCursor {
  int q, ls;      // piece, triple slot within the piece
  int64_t bt;     // block triple
  int64_t first;  // the block's first block triple of this triple
};

__device__ __forceinline__ int64_t cursor_first(const TcPiece& pc, int ls) {
  const int64_t r = ((int64_t)blockIdx.x - (pc.t0 + ls) * pc.nbt) % (int64_t)gridDim.x;
  return r < 0 ? r + gridDim.x : r;
}

__device__ __forceinline__ void cursor_settle(const EnergyParams& P, ItemCursor& c) {
  while (c.q < P.npieces) {
    const TcPiece& pc = P.pc[c.q];
    if (c.bt < 0) c.bt = c.first = cursor_first(pc, c.ls);
    if (c.bt < pc.nbt) return;
    c.bt = -1;  // no (more) items of this triple for this block
    if (++c.ls >= pc.ns) {
      c.ls = 0;
      ++c.q;
    }
  }
}

template <int CW>
__global__ void __launch_bounds__(THREADS, 1)
    k_energy_tc(const __grid_constant__ EnergyMaps M, const __grid_constant__ EnergyParams P) {
  using L = Layout<CW>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) &
                                                         ~uintptr_t(127));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + 2 * L::buf);    // [2]
  uint64_t* empty = full + 2;                                         // [2], one arrival per compute warp
  volatile int* abort_flag = reinterpret_cast<volatile int*>(empty + 2);
  int* meta = const_cast<int*>(reinterpret_cast<volatile int*>(abort_flag) + 1);  // [2][8]: X, Y, Z, slot, v, item

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int q = 0; q < 2; ++q) {
      ptx::mbar_init(&full[q], 2);  // the copies' arrive.expect_tx and the denominator table's arrive
      ptx::mbar_init(&empty[q], WARPS);
    }
    *abort_flag = 0;
    ptx::fence_barrier_init();
  }
  __syncthreads();

  if (warp == WARPS) {
    // ---------------- producer warp ----------------
    uint32_t ephase = 0u, pending = 0u, fphase = 0u;  // one bit per buffer
    int b = 0;
    bool ok = true;
    ItemCursor cur{0, 0, -1, -1};
    cursor_settle(P, cur);
    for (; ok && cur.q < P.npieces; cur.bt += gridDim.x, cursor_settle(P, cur), b ^= 1) {
      // buffer b free: all compute warps done with the item it held
      int good = 1;
      if (lane == 0) good = ptx::mbar_wait(&empty[b], ((ephase >> b) & 1u) ^ 1u, P.wait_ns) ? 1 : 0;
      good = __shfl_sync(0xffffffffu, good, 0);
      if (!good || *abort_flag) {
        if (lane == 0 && !*abort_flag) {
          *abort_flag = 1;
          if (atomicOr(P.err, ERR_WAIT_TIMEOUT) == 0) {
            P.err[1] = 11;
            P.err[2] = blockIdx.x;
          }
        }
        ok = false;
        break;
      }
      ephase ^= 1u << b;
      const TcPiece& pc = P.pc[cur.q];
      const EnergyCl& C = P.cl[pc.cl];
      const int slot = cur.ls;
      const int64_t bt = cur.bt;
      const int64_t local = (int64_t)slot * C.nbt + bt;
      int blk[3];
      decode_bt(bt, blk);
      const Triple tr = P.triples[pc.t0 + slot];
      unsigned char* base = smem + (size_t)b * L::buf;
      if (lane == 0) {
        meta[b * 8 + 0] = blk[0];
        meta[b * 8 + 1] = blk[1];
        meta[b * 8 + 2] = blk[2];
        meta[b * 8 + 3] = pc.slot0 + slot;
        meta[b * 8 + 4] = C.v;
        ptx::mbar_arrive_expect_tx(&full[b], L::tx);  // first of the two arrivals
        pending |= 1u << b;
      }
      __syncwarp();
      const CUtensorMap* map_ovs = &M.ovs[pc.cl];
      const CUtensorMap* map_t1 = &M.t1[pc.cl];
      for (int q = lane; q < 28; q += 32) {
        if (q == 0) {  // the item's 18 cubes, contiguous ([g][pid] as in shared memory)
          ptx::bulk_load(base, pc.gbuf + local * (18 * TB * TB * TB * CW), 18 * L::cube_bytes, &full[b]);
        } else if (q < 19) {
          // ovs block (pair, sx, sy) with sx != sy: the only ones a permutation's Y reads
          const int rr = q - 1, pair = rr / 6, od = rr % 6;
          const int sx = od >> 1, sy = (od == 0) ? 1 : (od == 1) ? 2 : (od == 2) ? 0 : (od == 3) ? 2 : (od == 4) ? 0 : 1;
          const int r = pair * 9 + sx * 3 + sy;
          const int P1 = (pair == 1) ? tr.j : tr.i;
          const int P2 = (pair == 0) ? tr.j : tr.k;
          ptx::tma_load_4d(base + L::cubes + r * 256, map_ovs, &full[b], blk[sy] * TB, P2, blk[sx] * TB, P1);
        } else {
          const int r = q - 19, which = r / 3, s2 = r % 3;
          const int occ = which == 0 ? tr.i : (which == 1 ? tr.j : tr.k);
          ptx::tma_load_2d(base + L::cubes + L::ovs + r * 128, map_t1, &full[b], blk[s2] * TB, occ);
        }
      }
      {  // FP64 denominator pieces while the copies fly: dAB[la][lb] = e_i+e_j+e_k - e_a - e_b, epsC[lc] = e_c
        // the 24 virtual energies of the three blocks, one load per lane, shared by shuffles
        double* dAB = reinterpret_cast<double*>(base + L::cubes + L::ovs + L::t1);
        const int lq = lane < 24 ? blk[lane >> 3] * TB + (lane & 7) : 0;
        const double ev = (lane < 24 && lq < C.v) ? C.eps_v[lq] : 0.0;
        const double eo = C.eps_o[tr.i] + C.eps_o[tr.j] + C.eps_o[tr.k];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          const int q = lane + 32 * r;  // every lane shuffles; lanes with q >= 72 store nothing
          const double ea = __shfl_sync(0xffffffffu, ev, q < 64 ? (q >> 3) : 16 + (q & 7));
          const double eb = __shfl_sync(0xffffffffu, ev, 8 + (q & 7));
          if (q < 64) {
            const int qa = blk[0] * TB + (q >> 3), qb = blk[1] * TB + (q & 7);
            dAB[q] = (qa < C.v && qb < C.v) ? (eo - ea) - eb : 0.0;
          } else if (q < 72) {
            const int qc = blk[2] * TB + (q - 64);
            dAB[q] = qc < C.v ? ea : 0.0;
          }
        }
      }
      __syncwarp();  // every lane's dAB stores are ordered before lane 0's release
      if (lane == 0) ptx::mbar_arrive(&full[b]);  // second arrival
      fphase ^= 1u << b;
    }
    // partials of the last items once their warps are done; copies in flight land
    if (lane == 0)
      for (int q = 0; q < 2; ++q)
        if (((pending >> q) & 1u) && !ok) ptx::mbar_wait(&full[q], ((fphase >> q) & 1u) ^ 1u, P.wait_ns);
  } else {
    // ---------------- compute warps ----------------
    // A thread takes the orbit (a,b,c) = its local point of the block triple.
    // With pid m a block order and A_m the same permutation of (la, lb, lc) in
    // cube m, W~ at position n is G0[A_n] + G1[A_r1(n)] + G2[A_r2(n)]: six
    // offsets address all 36 words, each read once, and no value crosses
    // threads.  (An earlier form assembled W~ and Y of the six orders in shared
    // memory first: 24 more stores and 18 more loads per thread, and two
    // block-wide barriers per item.)  The buffer goes back to the producer as
    // soon as the words are in registers.
    uint32_t phase = 0u;  // one bit per buffer
    int b = 0;
    const int la = (tid >> 6), lb = (tid >> 3) & 7, lc = tid & 7;
    int pos_off[6];
#pragma unroll
    for (int n = 0; n < 6; ++n) {
      const int u = n <= 1 ? la : (n <= 3 ? lb : lc);
      const int w = (n == 0 || n == 5) ? lb : ((n == 1 || n == 3) ? lc : la);
      const int z = (n == 0 || n == 2) ? lc : ((n == 1 || n == 4) ? lb : la);
      pos_off[n] = n * 512 * CW + cube_off(u, w, z);
    }
    // this thread's float64 sum over its items of the current triple slot; the
    // warp's sum (fixed shuffle order) goes to the partials when the slot
    // changes (a block takes a triple's items one after another)
    double acc = 0.0;
    int cur_slot = -1;
    int64_t cur_first = 0;
    auto flush = [&]() {
      double a = acc;
      for (int off = 16; off > 0; off >>= 1) a += __shfl_down_sync(0xffffffffu, a, off);
      if (lane == 0) P.partials[((int64_t)cur_slot * gridDim.x + cur_first) * WARPS + warp] = a;
      acc = 0.0;
    };
    ItemCursor cur{0, 0, -1, -1};
    cursor_settle(P, cur);
    for (; cur.q < P.npieces; cur.bt += gridDim.x, cursor_settle(P, cur), b ^= 1) {
      int got = 0;
      if (!*abort_flag) got = ptx::mbar_wait(&full[b], (phase >> b) & 1u, P.wait_ns) ? 1 : 0;
      if (!__all_sync(0xffffffffu, got)) {
        if (lane == 0 && !*abort_flag) {
          *abort_flag = 1;
          if (atomicOr(P.err, ERR_WAIT_TIMEOUT) == 0) {
            P.err[1] = 10;
            P.err[2] = blockIdx.x;
          }
        }
        break;
      }
      phase ^= 1u << b;
      const int bx = meta[b * 8 + 0], by = meta[b * 8 + 1], bz = meta[b * 8 + 2], slot = meta[b * 8 + 3];
      const int vcl = meta[b * 8 + 4];
      if (slot != cur_slot) {
        if (cur_slot >= 0) flush();
        cur_slot = slot;
        cur_first = cur.first;
      }
      const unsigned char* base = smem + (size_t)b * L::buf;
      const float* cube = reinterpret_cast<const float*>(base);
      const float* ovsS = reinterpret_cast<const float*>(base + L::cubes);
      const float* t1S = reinterpret_cast<const float*>(base + L::cubes + L::ovs);
      const double* dAB = reinterpret_cast<const double*>(base + L::cubes + L::ovs + L::t1);
      const double D = dAB[la * 8 + lb] - dAB[64 + lc];

      const int a = bx * TB + la, bb = by * TB + lb, c = bz * TB + lc;
      const bool valid = a < vcl && bb < vcl && c < vcl && !(bx == by && la < lb) && !(by == bz && lb < lc);
      float wh[6], wl[6], y[6];
      if (valid) {
        float t1v[3][3];  // [i, j, k][slot of the virtual]
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          t1v[q][0] = t1S[(q * 3 + 0) * 32 + la];
          t1v[q][1] = t1S[(q * 3 + 1) * 32 + lb];
          t1v[q][2] = t1S[(q * 3 + 2) * 32 + lc];
        }
#pragma unroll
        for (int n = 0; n < 6; ++n) {
          const int r1 = n == 0 ? 3 : n == 1 ? 5 : n == 2 ? 1 : n == 3 ? 4 : n == 4 ? 0 : 2;
          const int r2 = n == 0 ? 4 : n == 1 ? 2 : n == 2 ? 5 : n == 3 ? 0 : n == 4 ? 3 : 1;
          const int s0 = n <= 1 ? 0 : (n <= 3 ? 1 : 2);
          const int s1 = n == 0 ? 1 : n == 1 ? 2 : n == 2 ? 0 : n == 3 ? 2 : n == 4 ? 0 : 1;
          const int s2 = 3 - s0 - s1;
          const int x = s0 == 0 ? la : (s0 == 1 ? lb : lc), yy = s1 == 0 ? la : (s1 == 1 ? lb : lc),
                    z = s2 == 0 ? la : (s2 == 1 ? lb : lc);
          const float* g0 = cube + pos_off[n];
          const float* g1 = cube + 6 * 512 * CW + pos_off[r1];
          const float* g2 = cube + 12 * 512 * CW + pos_off[r2];
          if constexpr (CW == 2) {
            df wv = df_two_sum(g0[0], g1[0]);
            wv = df_add(wv, df{g2[0], 0.f});
            wv = df_norm(wv.h, __fadd_rn(wv.l, __fadd_rn(__fadd_rn(g0[512], g1[512]), g2[512])));
            wh[n] = wv.h;
            wl[n] = wv.l;
          } else {
            wh[n] = (g0[0] + g1[0]) + g2[0];
            wl[n] = 0.f;
          }
          // Y at (x, y, z) = positions (s0, s1, s2):
          //   ovs(i,x,j,y) t1(k,z) + ovs(j,y,k,z) t1(i,x) + ovs(i,x,k,z) t1(j,y)
          y[n] = fmaf(ovsS[((2 * 3 + s0) * 3 + s2) * 64 + x * 8 + z], t1v[1][s1],
                      fmaf(ovsS[((1 * 3 + s1) * 3 + s2) * 64 + yy * 8 + z], t1v[0][s0],
                           __fmul_rn(ovsS[((0 * 3 + s0) * 3 + s1) * 64 + x * 8 + yy], t1v[2][s2])));
        }
      }
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&empty[b]);  // this warp no longer reads buffer b
      if (valid) {
        // orbit weight A (Eq. E_corr_CCSD_T): 1, 1/2 or 1/6
        const bool all3 = (a == bb && bb == c), two = (a == bb || bb == c);
        const double r0 = (double)__frcp_rn((float)D);
        const double r1 = fma(r0, fma(-D, r0, 1.0), r0);  // 1/D to ~1e-14 (one Newton step)
        if constexpr (CW == 2) {
          df wd[5], vd[5];
#pragma unroll
          for (int n = 1; n < 6; ++n) {
            df d = df_two_sum(wh[n], -wh[0]);
            d = df_norm(d.h, __fadd_rn(d.l, __fsub_rn(wl[n], wl[0])));
            wd[n - 1] = d;
            vd[n - 1] = df_add(d, df{__fsub_rn(y[n], y[0]), 0.f});
          }
          const df w1 = wd[0], w2 = wd[1], w3 = wd[2], w4 = wd[3], w5 = wd[4];
          const df v1 = vd[0], v2 = vd[1], v3 = vd[2], v4 = vd[3], v5 = vd[4];
          const df Ae = df_add(w3, w4), Ao = df_add(df_add(w1, w2), w5);
          const df Se = df_add(v3, v4), So = df_add(df_add(v1, v2), v5);
          df dot = df_mul(w1, v1);
          dot = df_add(dot, df_mul(w2, v2));
          dot = df_add(dot, df_mul(w3, v3));
          dot = df_add(dot, df_mul(w4, v4));
          dot = df_add(dot, df_mul(w5, v5));
          df T = df_add(df_scale(dot, 3.f), df_add(df_mul(Ae, Se), df_mul(Ao, So)));
          T = df_add(T, df_scale(df_add(df_mul(Ae, So), df_mul(Ao, Se)), -2.f));
          if (all3) T = df_mul(T, df{0.16666667f, -4.967054e-09f});  // 1/6 as a float pair
          else if (two) T = df{T.h * 0.5f, T.l * 0.5f};
          acc = fma((double)T.h, r1, acc);
          acc = fma((double)T.l, r1, acc);
        } else {
          float w[5], vv[5];
#pragma unroll
          for (int n = 1; n < 6; ++n) {
            w[n - 1] = wh[n] - wh[0];
            vv[n - 1] = w[n - 1] + (y[n] - y[0]);
          }
          const float Ae = w[2] + w[3], Ao = w[0] + w[1] + w[4];
          const float Se = vv[2] + vv[3], So = vv[0] + vv[1] + vv[4];
          const float dot = w[0] * vv[0] + w[1] * vv[1] + w[2] * vv[2] + w[3] * vv[3] + w[4] * vv[4];
          const float T = 3.f * dot + Ae * Se + Ao * So - 2.f * (Ae * So + Ao * Se);
          const double Tw = all3 ? (double)T * (1.0 / 6.0) : (double)(two ? 0.5f * T : T);
          acc = fma(Tw, r1, acc);
        }
      }
    }
    if (cur_slot >= 0) flush();
  }
  __syncthreads();
}

}  // namespace

int64_t energy_tc_grid(int num_sms, int64_t items) {
  (void)items;  // one block per SM whatever the launch holds: the item-to-block map is fixed per triple
  return std::max(1, num_sms);
}

size_t energy_tc_smem(int cw) {
  const size_t buf = cw == 2 ? Layout<2>::buf : Layout<1>::buf;
  return 2 * buf + 128 + 512;
}

cudaError_t launch_energy_tc(const EnergyLaunch& e, cudaStream_t s) {
  EnergyMaps M;
  std::memset(&M, 0, sizeof(M));
  for (int c = 0; c < e.ncl; ++c) {
    M.ovs[c] = *e.map_ovs[c];
    M.t1[c] = *e.map_t1[c];
  }
  EnergyParams P;
  std::memset(&P, 0, sizeof(P));
  P.ncl = e.ncl;
  P.npieces = e.npieces;
  P.items = e.items;
  for (int c = 0; c < e.ncl; ++c) P.cl[c] = e.cl[c];
  for (int q = 0; q < e.npieces; ++q) P.pc[q] = e.pc[q];
  P.triples = e.triples;
  P.partials = e.partials;
  P.err = e.err;
  P.wait_ns = e.wait_ns;
  const size_t smem = energy_tc_smem(e.cw);
  const int64_t grid = energy_tc_grid(e.num_sms, P.items);
  cudaError_t err;
  if (e.cw == 2) {
    err = cudaFuncSetAttribute(k_energy_tc<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    k_energy_tc<2><<<(unsigned)grid, THREADS, smem, s>>>(M, P);
  } else {
    err = cudaFuncSetAttribute(k_energy_tc<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    k_energy_tc<1><<<(unsigned)grid, THREADS, smem, s>>>(M, P);
  }
  return cudaGetLastError();
}

// One block per slot: the partials of the blocks that took items of the triple
// (the first min(grid, nbt) x WARPS of the slot) summed in a fixed order
// (thread t takes t, t + 256, ..., then a fixed tree, with Neumaier
// compensation), times m/3, into its piece's shares.  A block is a chain of
// latencies (12 us for 2432 partials, whatever the launch holds), so one
// launch takes the slots of many rounds: at nocc=16 nvir=120, 200 launches of
// four slots were 2.5 ms of a 50 ms call.
__device__ __forceinline__ void neumaier(double& s, double& c, double x) {
  const double t = s + x;
  if (fabs(s) >= fabs(x)) c += (s - t) + x;
  else c += (x - t) + s;
  s = t;
}

__global__ void __launch_bounds__(256) k_reduce_pieces(const double* __restrict__ partials, int grid,
                                                       const Triple* __restrict__ triples,
                                                       const __grid_constant__ PieceTable T) {
  const int gslot = blockIdx.x;
  int q = 0;
  while (q + 1 < T.n && T.pc[q + 1].slot0 <= gslot) ++q;
  const TcPiece& pc = T.pc[q];
  const int local = gslot - pc.slot0;
  const int nper = (int)min((int64_t)grid, pc.nbt) * WARPS;
  const double* x = partials + (int64_t)gslot * grid * WARPS;
  __shared__ double ss[256], cc[256];
  double sum = 0.0, c = 0.0;
  for (int i = threadIdx.x; i < nper; i += blockDim.x) neumaier(sum, c, x[i]);
  ss[threadIdx.x] = sum;
  cc[threadIdx.x] = c;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) {
      double s1 = ss[threadIdx.x], c1 = cc[threadIdx.x] + cc[threadIdx.x + w];
      neumaier(s1, c1, ss[threadIdx.x + w]);
      ss[threadIdx.x] = s1;
      cc[threadIdx.x] = c1;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) pc.shares[local] = (ss[0] + cc[0]) * ((double)triples[pc.t0 + local].m / 3.0);
}

cudaError_t launch_reduce_pieces(const double* partials, int grid, const Triple* triples,
                                 const TcPiece* pieces, int npieces, int nslots, cudaStream_t s) {
  PieceTable T;
  std::memset(&T, 0, sizeof(T));
  T.n = npieces;
  for (int q = 0; q < npieces; ++q) T.pc[q] = pieces[q];
  k_reduce_pieces<<<(unsigned)nslots, 256, 0, s>>>(partials, grid, triples, T);
  return cudaGetLastError();
}

}  // namespace te
