// Energy epilogue of the tensor-core modes: a persistent kernel fed by TMA.
//
// Work item = (triple slot, block triple X >= Y >= Z of 8-wide virtual
// blocks).  The contraction kernel stores G orbit-major (energy_tc.h): the
// item's 18 G cubes (3 G blocks x 6 block orders) are contiguous and arrive
// by one bulk copy; the 18 8x8 blocks of the symmetrised ovov the item uses
// and 9 t1 rows come by TMA (few, large copies: the copy engine's per-copy
// cost, not HBM, limited a layout that needed 54 copies per item).  A ring of
// two to four buffers has a producer warp each: an item's decode, its loads of
// the triple and the orbital energies and its float64 table are one chain of
// some thousand cycles, which a single producer could not keep ahead of the
// sixteen compute warps.  One thread per orbit candidate (a,b,c) of the 8^3
// block triple.
//
// Orbit sum.  R's coefficient pattern between the six orbit positions has zero
// row and column sums, so only differences of W~ enter, and the symmetric part
// of W~, which R annihilates, never enters a rounded product.  With the even
// positions e = (0, 3, 4), the odd ones o = (1, 2, 5), d1 = w_e0 - w_e1,
// d2 = w_e1 - w_e2 (o alike), d' the same of V = W~ + Y, and X, X' the sums over
// the even positions less those over the odd ones:
//   T = sum_{e,o} [d1 (2 d1' + d2') + d2 (d1' + 2 d2')] + 2 X X',
// five products (the form 3 sum w v + Ae Se + Ao So - 2 (Ae So + Ao Se) over the
// deviations from position 0 takes nine).  W~, the differences and the products
// are FP32 pairs whose high parts are summed without error (two-sum,
// two-product) and whose low parts collect the rest.  D, its reciprocal (FP32
// seed + one Newton step in FP64: error ~1e-14), A T / D and the sums are FP64.
#include <cstring>

#include "energy_tc.h"
#include "fp_util.cuh"
#include "ptx_sm100.cuh"

namespace te {

namespace {

constexpr int TB = 8;
constexpr int WARPS = 16;                 // compute warps: one orbit candidate (a,b,c) of 8^3 per thread

template <int FMT>
struct Layout {
  static constexpr uint32_t cube_bytes = g_cube_floats(FMT) * 4;
  static constexpr uint32_t cubes = 18 * cube_bytes;
  static constexpr uint32_t ovs = 27 * TB * TB * 4;
  static constexpr uint32_t t1 = 9 * 128;
  static constexpr uint32_t eps = 640;  // dAB[64] = e_ijk - e_a - e_b, epsC[8] (FP64, written by the producer)
  static constexpr uint32_t buf = cubes + ovs + t1 + eps;
  // A consumer holds a buffer for most of an item's arithmetic, and a copy
  // takes about as long: two buffers left the warps waiting for half the time
  // at nvir = 320.  As many as 227 KB hold, at most four.
  static constexpr int nbuf = FMT == G_F32 ? 4 : (FMT == G_PAIR ? 2 : 3);
  static constexpr uint32_t tx = 18 * cube_bytes + 18 * TB * TB * 4 + 9 * TB * 4;
  static constexpr size_t smem = (size_t)nbuf * buf + 128 + 512;
  static constexpr int threads = (WARPS + nbuf) * 32;  // one producer warp per buffer
};
static_assert(Layout<G_F32>::smem <= 227 * 1024 && Layout<G_PAIR>::smem <= 227 * 1024 &&
                  Layout<G_MIXED>::smem <= 227 * 1024, "shared memory of one block");

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

// ---- pairs of FP32 (value h + l): error-free transformations ----
// Knuth two-sum, FMA two-product; the rn intrinsics forbid contraction.  W~
// and its differences are renormalised, |l| <= ulp(h) / 2, after every
// operation: where R annihilates most of W~ the high parts cancel, and a low
// part left as large as what remains of them would cut the products that
// follow to 24 + 8 bits (W~ 2^15 times its differences: 4e-13 of a share
// against 1e-15).  Sums of products and of FP32 terms stay as they come.
struct df {
  float h, l;
};

__device__ __forceinline__ df two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}

__device__ __forceinline__ df df_norm(float h, float l) {
  const float s = __fadd_rn(h, l);
  return {s, __fsub_rn(l, __fsub_rn(s, h))};
}

__device__ __forceinline__ df df_add(df a, df b) {
  const df s = two_sum(a.h, b.h);
  return df_norm(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}

__device__ __forceinline__ df df_sub(df a, df b) { return df_add(a, df{-b.h, -b.l}); }

__device__ __forceinline__ df df_addf(df a, float b) {
  const df s = two_sum(a.h, b);
  return {s.h, __fadd_rn(s.l, a.l)};
}

// acc += a b
__device__ __forceinline__ void df_fma(df& acc, df a, df b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = fmaf(a.h, b.h, -p);
  e = fmaf(a.h, b.l, e);
  e = fmaf(a.l, b.h, e);
  e = fmaf(a.l, b.l, e);
  const df s = two_sum(acc.h, p);
  acc.h = s.h;
  acc.l = __fadd_rn(acc.l, __fadd_rn(s.l, e));
}

// 2 a + b
__device__ __forceinline__ df df_2ab(df a, df b) {
  const df s = two_sum(2.f * a.h, b.h);
  return {s.h, __fadd_rn(s.l, __fadd_rn(2.f * a.l, b.l))};
}

struct EnergyMaps {
  CUtensorMap ovs[TC_MAX_CL];  // per cluster: ovs32 [o][v][o][vq], 4D (b, j, a, i)
  CUtensorMap t1[TC_MAX_CL];   // per cluster: t1 [o][vq], 2D (a, i)
};

struct EnergyParams {
  int npieces;
  EnergyCl cl[TC_MAX_CL];
  TcPiece pc[TC_MAX_PIECES];  // G: orbit-major [slot][bt][g][pid][cube] from pc.gbuf
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

// Bound by instruction issue (60% of cycles; float64 pipe and HBM 44% each).
// nocc=32 nvir=320: 185 us per triple (177 without the renormalisations); 272 us with the assembled area, 8-byte G
// and one producer warp, 240 us with one producer for three buffers.
template <int FMT>
__global__ void __launch_bounds__(Layout<FMT>::threads, 1)
    k_energy_tc(const __grid_constant__ EnergyMaps M, const __grid_constant__ EnergyParams P) {
  using L = Layout<FMT>;
  constexpr int NB = L::nbuf, CUBE = g_cube_floats(FMT);
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) &
                                                         ~uintptr_t(127));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + NB * L::buf);  // [NB]
  uint64_t* empty = full + NB;                                       // [NB], one arrival per compute warp
  volatile int* abort_flag = reinterpret_cast<volatile int*>(empty + NB);
  int* meta = const_cast<int*>(reinterpret_cast<volatile int*>(abort_flag) + 1);  // [NB][8]: X, Y, Z, slot, v

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int q = 0; q < NB; ++q) {
      ptx::mbar_init(&full[q], 2);  // the copies' arrive.expect_tx and the denominator table's arrive
      ptx::mbar_init(&empty[q], WARPS);
    }
    *abort_flag = 0;
    ptx::fence_barrier_init();
  }
  __syncthreads();

  if (warp >= WARPS) {
    // ---------------- producer warps: buffer b = every NB-th item ----------------
    const int b = warp - WARPS;
    uint32_t ph = 0u;  // parity of the ring's current turn
    int at = 0;        // buffer of the cursor's item
    bool ok = true, issued = false;
    ItemCursor cur{0, 0, -1, -1};
    cursor_settle(P, cur);
    for (; ok && cur.q < P.npieces; cur.bt += gridDim.x, cursor_settle(P, cur), at = at + 1 == NB ? 0 : at + 1) {
      if (at != b) continue;
      const TcPiece& pc = P.pc[cur.q];
      const EnergyCl& C = P.cl[pc.cl];
      const int slot = cur.ls;
      const int64_t bt = cur.bt;
      const int64_t local = (int64_t)slot * C.nbt + bt;
      int blk[3];
      decode_bt(bt, blk);
      // the loads that the item's table needs, before the wait for its buffer:
      // the 24 virtual energies of the three blocks, one per lane
      const Triple tr = P.triples[pc.t0 + slot];
      const int lq = lane < 24 ? blk[lane >> 3] * TB + (lane & 7) : 0;
      const double ev = (lane < 24 && lq < C.v) ? C.eps_v[lq] : 0.0;
      const double eo = C.eps_o[tr.i] + C.eps_o[tr.j] + C.eps_o[tr.k];
      // buffer b free: all compute warps done with the item it held
      int good = 1;
      if (lane == 0) good = ptx::mbar_wait(&empty[b], ph ^ 1u, P.wait_ns) ? 1 : 0;
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
      unsigned char* base = smem + (size_t)b * L::buf;
      if (lane == 0) {
        meta[b * 8 + 0] = blk[0];
        meta[b * 8 + 1] = blk[1];
        meta[b * 8 + 2] = blk[2];
        meta[b * 8 + 3] = pc.slot0 + slot;
        meta[b * 8 + 4] = C.v;
        ptx::mbar_arrive_expect_tx(&full[b], L::tx);  // first of the two arrivals
      }
      __syncwarp();
      const CUtensorMap* map_ovs = &M.ovs[pc.cl];
      const CUtensorMap* map_t1 = &M.t1[pc.cl];
      if (lane == 0) {  // the item's 18 cubes, contiguous ([g][pid] as in shared memory)
        ptx::bulk_load(base, pc.gbuf + local * (18 * CUBE), 18 * L::cube_bytes, &full[b]);
      } else if (lane < 19) {
        // ovs block (pair, sx, sy) with sx != sy: the only ones a permutation's Y reads
        const int rr = lane - 1, pair = rr / 6, od = rr % 6;
        const int sx = od >> 1, sy = (od == 0) ? 1 : (od == 1) ? 2 : (od == 2) ? 0 : (od == 3) ? 2 : (od == 4) ? 0 : 1;
        const int r = pair * 9 + sx * 3 + sy;
        const int P1 = (pair == 1) ? tr.j : tr.i;
        const int P2 = (pair == 0) ? tr.j : tr.k;
        ptx::tma_load_4d(base + L::cubes + r * 256, map_ovs, &full[b], blk[sy] * TB, P2, blk[sx] * TB, P1);
      } else if (lane < 28) {
        const int r = lane - 19, which = r / 3, s2 = r % 3;
        const int occ = which == 0 ? tr.i : (which == 1 ? tr.j : tr.k);
        ptx::tma_load_2d(base + L::cubes + L::ovs + r * 128, map_t1, &full[b], blk[s2] * TB, occ);
      }
      __syncwarp();
      {  // FP64 denominator pieces while the copies fly: dAB[la][lb] = e_i+e_j+e_k - e_a - e_b, epsC[lc] = e_c
        double* dAB = reinterpret_cast<double*>(base + L::cubes + L::ovs + L::t1);
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
      issued = true;
      ph ^= 1u;
    }
    // The copies of this buffer's last item land before the block ends.  The
    // consumers wait for them only as long as none of their waits has expired,
    // which this warp's own loop need not have seen.
    if (lane == 0 && issued) ptx::mbar_wait(&full[b], ph ^ 1u, P.wait_ns);
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
    uint32_t ph = 0u;
    int b = 0;
    const int la = (tid >> 6), lb = (tid >> 3) & 7, lc = tid & 7;
    int pos_off[6];
#pragma unroll
    for (int n = 0; n < 6; ++n) {
      const int u = n <= 1 ? la : (n <= 3 ? lb : lc);
      const int w = (n == 0 || n == 5) ? lb : ((n == 1 || n == 3) ? lc : la);
      const int z = (n == 0 || n == 2) ? lc : ((n == 1 || n == 4) ? lb : la);
      pos_off[n] = cube_off(u, w, z);
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
    for (; cur.q < P.npieces; cur.bt += gridDim.x, cursor_settle(P, cur)) {
      int got = 0;
      if (!*abort_flag) got = ptx::mbar_wait(&full[b], ph, P.wait_ns) ? 1 : 0;
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
      const int a = bx * TB + la, bb = by * TB + lb, c = bz * TB + lc;
      const bool valid = a < vcl && bb < vcl && c < vcl && !(bx == by && la < lb) && !(by == bz && lb < lc);
      df w[6];
      float y[6];
      double D = 0.0;
      if (valid) {
        D = dAB[la * 8 + lb] - dAB[64 + lc];
        // plane word(s) of G block g at pid m
        auto gv = [&](int g, int m) -> df {
          const float* p = cube + (g * 6 + m) * CUBE;
          if constexpr (FMT == G_PAIR) return {p[pos_off[m]], p[512 + pos_off[m]]};
          if constexpr (FMT == G_MIXED)
            return {p[pos_off[m]],
                    __uint_as_float((uint32_t)reinterpret_cast<const unsigned short*>(p + 512)[pos_off[m]] << 16)};
          return {p[pos_off[m]], 0.f};
        };
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
          const df g0 = gv(0, n), g1 = gv(1, r1), g2 = gv(2, r2);
          if constexpr (FMT == G_F32) {
            w[n] = df{(g0.h + g1.h) + g2.h, 0.f};
          } else {
            const df s = two_sum(g0.h, g1.h), s3 = two_sum(s.h, g2.h);
            w[n] = df_norm(s3.h, __fadd_rn(__fadd_rn(s.l, s3.l), __fadd_rn(__fadd_rn(g0.l, g1.l), g2.l)));
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
      if (++b == NB) {
        b = 0;
        ph ^= 1u;
      }
      if (valid) {
        // orbit weight A (Eq. E_corr_CCSD_T): 1, 1/2 or 1/6
        const bool all3 = (a == bb && bb == c), two = (a == bb || bb == c);
        const double r1 = recip_newton(D, recip_seed(D));
        if constexpr (FMT != G_F32) {
          // differences of W~ within the even (0, 3, 4) and odd (1, 2, 5) positions, and even less odd
          const df e1 = df_sub(w[0], w[3]), e2 = df_sub(w[3], w[4]);
          const df o1 = df_sub(w[1], w[2]), o2 = df_sub(w[2], w[5]);
          const df X = df_add(df_add(df_sub(w[0], w[1]), df_sub(w[3], w[2])), df_sub(w[4], w[5]));
          // the same of V = W~ + Y
          const df fe1 = df_addf(e1, __fsub_rn(y[0], y[3])), fe2 = df_addf(e2, __fsub_rn(y[3], y[4]));
          const df fo1 = df_addf(o1, __fsub_rn(y[1], y[2])), fo2 = df_addf(o2, __fsub_rn(y[2], y[5]));
          const df S = df_addf(df_addf(df_addf(X, __fsub_rn(y[0], y[1])), __fsub_rn(y[3], y[2])), __fsub_rn(y[4], y[5]));
          df t{0.f, 0.f};
          df_fma(t, X, df{2.f * S.h, 2.f * S.l});
          df_fma(t, e1, df_2ab(fe1, fe2));
          df_fma(t, e2, df_2ab(fe2, fe1));
          df_fma(t, o1, df_2ab(fo1, fo2));
          df_fma(t, o2, df_2ab(fo2, fo1));
          df T = df_norm(t.h, t.l);
          if (two) {
            const float k = all3 ? 0.16666667f : 0.5f, kl = all3 ? -4.967054e-09f : 0.f;  // 1/6 as a float pair
            const float p = __fmul_rn(T.h, k);
            T = df_norm(p, fmaf(T.l, k, fmaf(T.h, kl, fmaf(T.h, k, -p))));
          }
          acc = fma(to_double(T.h), r1, acc);
          acc = fma(to_double(T.l), r1, acc);
        } else {
          float d[5], vv[5];
#pragma unroll
          for (int n = 1; n < 6; ++n) {
            d[n - 1] = w[n].h - w[0].h;
            vv[n - 1] = d[n - 1] + (y[n] - y[0]);
          }
          const float Ae = d[2] + d[3], Ao = d[0] + d[1] + d[4];
          const float Se = vv[2] + vv[3], So = vv[0] + vv[1] + vv[4];
          const float dot = d[0] * vv[0] + d[1] * vv[1] + d[2] * vv[2] + d[3] * vv[3] + d[4] * vv[4];
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

// one block per SM whatever the launch holds: the item-to-block map is fixed per triple
int64_t energy_tc_grid(int num_sms) { return std::max(1, num_sms); }

template <int FMT>
static cudaError_t launch_fmt(const EnergyMaps& M, const EnergyParams& P, int64_t grid, cudaStream_t s) {
  constexpr size_t smem = Layout<FMT>::smem;
  const cudaError_t e = cudaFuncSetAttribute(k_energy_tc<FMT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_energy_tc<FMT><<<(unsigned)grid, Layout<FMT>::threads, smem, s>>>(M, P);
  return cudaGetLastError();
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
  P.npieces = e.npieces;
  for (int c = 0; c < e.ncl; ++c) P.cl[c] = e.cl[c];
  for (int q = 0; q < e.npieces; ++q) P.pc[q] = e.pc[q];
  P.triples = e.triples;
  P.partials = e.partials;
  P.err = e.err;
  P.wait_ns = e.wait_ns;
  const int64_t grid = energy_tc_grid(e.num_sms);
  if (e.fmt == G_MIXED) return launch_fmt<G_MIXED>(M, P, grid, s);
  if (e.fmt == G_PAIR) return launch_fmt<G_PAIR>(M, P, grid, s);
  return launch_fmt<G_F32>(M, P, grid, s);
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
