// Exact-slice contractions on tcgen05 over tensor-map views (see view_tc.h).
//
// Warp roles of the persistent kernel: warp 0 issues the TMA copies (one
// five-dimensional box per operand and stage, all slices in it), warp 1 issues
// tcgen05.mma into three FP32 accumulators in tensor memory (the whole warp in
// step, one elected lane: the operands then sit in uniform registers; issued
// from a single-thread branch an MMA took 75 to 80 cycles whatever its size),
// warps 2..9 (two per TMEM lane quarter, half of the N tile each) drain every
// accumulation block into an FP32 pair sum held in registers and release the
// accumulators at once, so the next block's MMAs overlap the rest of the
// epilogue.  A unit's sum leaves once,
// at its end, converted to float64 by integer operations (GB300's float64 rate is
// a small fraction of its FP32 rate: two float64 operations per element took 12 of
// 30 thousand cycles of a 128 x 64 unit with four blocks).
//
// On CTA pairs an N tile of at most 64 leaves room for the accumulators of two
// blocks: the next block's MMAs run while the last one is drained.  What bounds
// the short-K launches then is tensor memory, whose loads and the MMAs' sums
// share its ports: a drain takes 2300 cycles alone and 3300 beside MMAs, and
// neither 16 epilogue warps nor a sum of four instructions changes it much.
// Eight triples of a gradient at nvir = 120, one set of 128 columns -> two of 64:
// G 671 -> 520 us, ovvv and t2 479 -> 384; one triple at nvir = 320: 1981 -> 1561,
// 2057 -> 1503.  The projected energy's pairs, which convert nothing, gain nothing
// from it (1096 -> 1105); one rule serves all.
// Lone CTAs have K of nvir^2: few drains, so one set of 128 columns, whose operands
// from L2 bound them (tensor pipe 49% active at nvir = 320).
//
// Pairs of CTAs share a B tile (cta_group::2): each loads its 128 A rows and half
// of B, rank 0 issues the MMAs of both SMs, and all bytes of the pair count on
// rank 0's barriers; the release of a stage and of the accumulators goes to both
// CTAs.
// Shared memory per stage: the A slices (128 rows of 64 bytes each, 64-byte
// swizzle, K-major) then this CTA's B rows of every slice.  Every wait is
// bounded; on expiry the kernel records the error word and unwinds.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>
#include <memory>
#include <new>

#include "fp_util.cuh"
#include "ptx_sm100.cuh"
#include "tc_path.h"
#include "view_tc.h"

namespace te {

namespace {

constexpr int VT_EPI_WARPS = 8;
constexpr int VT_WARPS = 2 + VT_EPI_WARPS;
constexpr int VT_THREADS = VT_WARPS * 32;
constexpr uint32_t VT_ROW_BYTES = VT_KC * 2;         // 64
constexpr uint32_t VT_A_SLICE = 128u * VT_ROW_BYTES;  // 8 KB

struct VtUnit {
  int job, split, m, n0;
  int64_t b_begin, b_end;
};

// unit u; m: the m tile of CTA `rank` (PAIR: of the unit's two); j: the job of a
// unit before it
template <bool PAIR>
__device__ __forceinline__ VtUnit vt_decode(const VtParams& P, int64_t u, int rank, int j) {
  VtUnit U;
  while (j + 1 < P.njobs && P.job[j + 1].unit0 <= u) ++j;
  const VtJob& J = P.job[j];
  uint32_t l = (uint32_t)(u - J.unit0);
  U.job = j;
  U.split = (int)(l % (uint32_t)J.nsplit);
  l /= (uint32_t)J.nsplit;
  const uint32_t mu = l / (uint32_t)J.nn;
  U.n0 = (int)(l - mu * (uint32_t)J.nn) * J.NT;
  U.m = PAIR ? 2 * (int)mu + rank : (int)mu;
  U.b_begin = J.nblocks * U.split / J.nsplit;
  U.b_end = J.nblocks * (U.split + 1) / J.nsplit;
  return U;
}

// accumulation blocks of a unit, in order
struct VtBlock {
  int seg, c0, c1;  // segment (in VtParams::seg) and its chunk range
};
__device__ __forceinline__ VtBlock vt_first(const VtParams& P, const VtJob& J, int64_t b) {
  int s = J.seg0;
  for (;;) {
    const int nblk = (P.seg[s].nchunks + J.bchunks - 1) / J.bchunks;
    if (b < nblk) break;
    b -= nblk;
    ++s;
  }
  const int c0 = (int)b * J.bchunks;
  return VtBlock{s, c0, min(c0 + J.bchunks, P.seg[s].nchunks)};
}
__device__ __forceinline__ void vt_next(const VtParams& P, const VtJob& J, VtBlock& B) {
  if (B.c1 < P.seg[B.seg].nchunks) {
    B.c0 = B.c1;
  } else {
    ++B.seg;
    B.c0 = 0;
    if (B.seg >= J.seg0 + J.nseg) return;  // past the last block
  }
  B.c1 = min(B.c0 + J.bchunks, P.seg[B.seg].nchunks);
}

template <bool PAIR>
__device__ __forceinline__ void vt_load(void* dst, const CUtensorMap* map, const VtRoles& R, const int16_t* fix,
                                        int kc, int r2, int r1, int k1, uint64_t* own, uint32_t bar) {
  int c[5];
#pragma unroll
  for (int d = 0; d < 5; ++d) {
    int x = d >= 2 ? fix[d - 2] : 0;
    if (d == R.k2) x = kc;
    if (d == R.r2) x = r2;
    if (d == R.r1) x = r1;
    if (d == R.k1) x = k1;
    if (d == R.s) x = 0;
    c[d] = x;
  }
  if (PAIR) ptx::tma_load_5d_pair(dst, map, bar, c[0], c[1], c[2], c[3], c[4]);
  else ptx::tma_load_5d(dst, map, own, c[0], c[1], c[2], c[3], c[4]);
}

__device__ __forceinline__ void vt_abort(const VtParams& P, volatile int* abort_flag, unsigned site) {
  *abort_flag = 1;
  if (atomicOr(P.err, ERR_WAIT_TIMEOUT) == 0) {
    P.err[1] = site;
    P.err[2] = blockIdx.x;
  }
}

template <bool PAIR>
__device__ __forceinline__ void vt_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  if (PAIR) ptx::mma_pair<false>(d, a, b, idesc, acc);
  else ptx::mma<false>(d, a, b, idesc, acc);
}
template <bool PAIR>
__device__ __forceinline__ void vt_mma_acc(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc) {
  if (PAIR) ptx::mma_acc_pair<false>(d, a, b, idesc);
  else ptx::mma_acc<false>(d, a, b, idesc);
}
template <bool PAIR>
__device__ __forceinline__ void vt_commit(uint64_t* bar) {
  if (PAIR) ptx::mma_commit_pair(bar);
  else ptx::mma_commit(bar);
}

// How a block joins the unit's sum (view_tc.h), two columns per packed
// instruction: a0 and a1, the exact FP32 sums of levels 0 and 1, a2 the rest, w a
// power of two.  These instructions sit between two blocks' MMAs, so each output
// kind pays for the precision it needs: VT_STORE 20, VT_PAIR 17, VT_ADD 23.
template <int SUM>
__device__ __forceinline__ void join(f2& H, f2& L, f2 a0, f2 a1, f2 a2, f2 w) {
  f2 s0, e0, t, te;
  f2_two_sum(a0, a1, s0, e0);
  const f2 x = f2_mul(s0, w), y = f2_mul(f2_add(e0, a2), w);
  f2_two_sum(H, x, t, te);
  if constexpr (SUM == VT_STORE) {
    const f2 l = f2_add(te, f2_add(L, y));
    H = f2_add(t, l);
    L = f2_sub(l, f2_sub(H, t));
  } else if constexpr (SUM == VT_PAIR) {
    H = t;
    L = f2_add(L, f2_add(te, y));
  } else {  // y can be 2^-14 of the operands' scale, far above the last bits of L: added without error
    f2 ye;
    f2_two_sum(t, y, H, ye);
    L = f2_add(L, f2_add(te, ye));
  }
}

// SUM: the output kind of every job of the launch.
template <int NS, bool PAIR, int SUM>
__device__ __forceinline__ void view_tc_body(const VtMaps& maps, const VtParams& P) {
  constexpr int SETS = PAIR ? 2 : 1;  // sets of accumulators
  constexpr int COLS = (PAIR ? VT_NT_PAIR : VT_NT_MAX) / 2;  // columns an epilogue thread holds at most
  constexpr int LD = PAIR ? 16 : 8;                          // and reads at once
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                         ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + (size_t)P.stages * P.stage_bytes);
  uint64_t* empty = full + P.stages;
  uint64_t* tfull = empty + P.stages;
  uint64_t* tempty = tfull + SETS;
  uint64_t* drain = tempty + SETS;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  constexpr int W = PAIR ? 2 : 1;  // CTAs per unit
  const int rank = PAIR ? (int)ptx::cluster_ctarank() : 0;
  const int64_t u0 = blockIdx.x / W, ustep = gridDim.x / W;
  if (threadIdx.x == 0) {
    for (int s = 0; s < P.stages; ++s) {
      ptx::mbar_init(&full[s], 1);
      ptx::mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < SETS; ++a) {
      ptx::mbar_init(&tfull[a], 1);
      ptx::mbar_init(&tempty[a], W * VT_EPI_WARPS);
    }
    ptx::mbar_init(drain, 1);
    *abort_flag = 0;
    ptx::fence_barrier_init();
  }
  // the scale exponents of all segments, read once
  __shared__ int seg_exp[VT_MAX_SEGS];
  for (int q = threadIdx.x; q < P.nsegs; q += VT_THREADS) seg_exp[q] = *P.seg[q].ea + *P.seg[q].eb;
  if (warp == 1) {
    if (PAIR) {
      ptx::tmem_alloc_pair(tmem_slot, P.tmem_cols);
      ptx::tmem_relinquish_pair();
    } else {
      ptx::tmem_alloc(tmem_slot, P.tmem_cols);
      ptx::tmem_relinquish();
    }
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (PAIR) ptx::cluster_sync();  // the barriers of both CTAs are initialised before either is signalled
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      uint32_t stage = 0, phase = 0;
      int pending[8];
      for (int s = 0; s < 8; ++s) pending[s] = -1;
      bool ok = true;
      int jq = 0;
      for (int64_t u = u0; ok && u < P.total_units; u += ustep) {
        const VtUnit U = vt_decode<PAIR>(P, u, rank, jq);
        jq = U.job;
        const VtJob& J = P.job[U.job];
        // the second tile of an odd last pair lies beyond the rows: its loads fill zeros
        const int m1t = U.m / J.nm2, m1_0 = m1t * J.TA, m2_0 = (U.m - m1t * J.nm2) * J.TB;
        const int br = PAIR ? U.n0 + rank * (J.NT / 2) : U.n0;
        const uint32_t bytes = (uint32_t)NS * (W * VT_A_SLICE + (uint32_t)J.NT * VT_ROW_BYTES);
        VtBlock B = vt_first(P, J, U.b_begin);
        for (int64_t b = U.b_begin; ok && b < U.b_end; ++b) {
          const VtSeg& S = P.seg[B.seg];
          const VtRoles& RA = P.roles[S.amap];
          const VtRoles& RB = P.roles[S.bmap];
          int k1 = B.c0 / S.nk2c, k2c = B.c0 - k1 * S.nk2c;
          for (int c = B.c0; c < B.c1; ++c) {
            if (*abort_flag || !ptx::mbar_wait(&empty[stage], phase ^ 1u, P.wait_ns)) {
              if (!*abort_flag) vt_abort(P, abort_flag, 21);
              ok = false;
              break;
            }
            if (rank == 0) ptx::mbar_arrive_expect_tx(&full[stage], bytes);
            const uint32_t bar = PAIR ? ptx::mapa(&full[stage], 0) : 0u;
            pending[stage] = (int)phase;
            unsigned char* sa = smem + (size_t)stage * P.stage_bytes;
            unsigned char* sb = sa + NS * VT_A_SLICE;
            vt_load<PAIR>(sa, &maps.m[S.amap], RA, S.afix, k2c * VT_KC, m2_0, m1_0, k1, &full[stage], bar);
            vt_load<PAIR>(sb, &maps.m[S.bmap], RB, S.bfix, k2c * VT_KC, br, 0, k1, &full[stage], bar);
            if (++k2c == S.nk2c) {
              k2c = 0;
              ++k1;
            }
            if (++stage == (uint32_t)P.stages) {
              stage = 0;
              phase ^= 1u;
            }
          }
          vt_next(P, J, B);
        }
      }
      // Before the CTA (or pair) exits: the MMAs have released every stage, so
      // every copy has landed too.  After an expired wait they may not come:
      // rank 0 waits for the copies it expects, and both for longer than a
      // copy takes.
      for (int s = 0; s < P.stages; ++s) {
        if (pending[s] < 0) continue;
        if (ok && !*abort_flag) ptx::mbar_wait(&empty[s], (uint32_t)pending[s], P.wait_ns);
        else if (rank == 0) ptx::mbar_wait(&full[s], (uint32_t)pending[s], P.wait_ns);
      }
      if (!ok || *abort_flag) ptx::pause_ns(200000);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (rank 0) ----------------
    uint32_t stage = 0, phase = 0, acc = 0, acc_phase = 0;
    bool ok = true, issued = false;
    auto wait_all = [&](uint64_t* bar, uint32_t parity, unsigned site) -> bool {
      const int got = (!*abort_flag && ptx::mbar_wait(bar, parity, P.wait_ns)) ? 1 : 0;
      const bool all = __all_sync(0xffffffffu, got);
      if (!all && lane == 0 && !*abort_flag) vt_abort(P, abort_flag, site);
      return all;
    };
    const uint32_t smem0 = ptx::smem_u32(smem);
    const uint64_t desc0 = ptx::smem_desc(0, 8u * VT_ROW_BYTES, 4u);  // 8 rows of the 64-byte swizzle
    int jq = 0;
    for (int64_t u = u0; ok && rank == 0 && u < P.total_units; u += ustep) {
      const VtUnit U = vt_decode<PAIR>(P, u, 0, jq);
      jq = U.job;
      const VtJob& J = P.job[U.job];
      const uint32_t NT = (uint32_t)J.NT;
      // kind::f16, BF16 A and B (K-major), FP32 accumulation, M = 128 or 256, N = NT
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((NT >> 3) << 17) |
                             ((uint32_t)(W * 128 >> 4) << 24);
      const uint32_t bstep = (NT / W) * VT_ROW_BYTES >> 4;
      VtBlock B = vt_first(P, J, U.b_begin);
      for (int64_t b = U.b_begin; ok && b < U.b_end; ++b) {
        const uint32_t d0 = tmem_base + acc * 3u * (uint32_t)P.nt_max, d1 = d0 + NT, dr = d1 + NT;
        if (!wait_all(&tempty[acc], acc_phase ^ 1u, 22)) {
          ok = false;
          break;
        }
        ptx::tc_fence_after();
        uint32_t first = 1;
        for (int c = B.c0; c < B.c1; ++c) {
          if (!wait_all(&full[stage], phase, 23)) {
            ok = false;
            break;
          }
          ptx::tc_fence_after();
          const uint32_t a0 = (smem0 + stage * P.stage_bytes) >> 4;
          const uint32_t b0 = a0 + (NS * VT_A_SLICE >> 4);
#pragma unroll
          for (int ks = 0; ks < VT_KC / 16; ++ks) {
            uint64_t ad[NS], bd[NS];
#pragma unroll
            for (int k = 0; k < NS; ++k) {
              ad[k] = desc0 + (a0 + k * (VT_A_SLICE >> 4) + ks * 2);
              bd[k] = desc0 + (b0 + k * bstep + ks * 2);
            }
            // slice products a_i b_j, i + j <= NS - 1: level 0 and level 1 in
            // their own (exact) accumulators, the higher levels in a third
            const uint32_t acc_in = first ? 0u : 1u;
            if (ptx::elect_one()) {
              vt_mma<PAIR>(d0, ad[0], bd[0], idesc, acc_in);
              vt_mma<PAIR>(d1, ad[0], bd[1], idesc, acc_in);
              vt_mma_acc<PAIR>(d1, ad[1], bd[0], idesc);
              vt_mma<PAIR>(dr, ad[0], bd[2], idesc, acc_in);
#pragma unroll
              for (int lev = 2; lev < NS; ++lev)
#pragma unroll
                for (int i = lev == 2 ? 1 : 0; i <= lev; ++i) vt_mma_acc<PAIR>(dr, ad[i], bd[lev - i], idesc);
            }
            first = 0;
          }
          issued = true;
          if (ptx::elect_one()) vt_commit<PAIR>(&empty[stage]);
          if (++stage == (uint32_t)P.stages) {
            stage = 0;
            phase ^= 1u;
          }
        }
        if (!ok) break;
        if (ptx::elect_one()) vt_commit<PAIR>(&tfull[acc]);
        if (++acc == SETS) {
          acc = 0;
          acc_phase ^= 1u;
        }
        vt_next(P, J, B);
      }
    }
    // every issued MMA completes before TMEM is released
    if (issued) {
      if (ptx::elect_one()) {
        if (PAIR) ptx::mma_commit_pair_own(drain);
        else ptx::mma_commit(drain);
      }
      ptx::mbar_wait(drain, 0, P.wait_ns);
    }
    __syncwarp();
  } else {
    // ---------------- epilogue: TMEM -> double-float -> output ----------------
    const int quad = warp & 3;               // the lane quarter this warp may read
    const int half = (warp - 2) >> 2;        // which half of the N tile
    const int row = quad * 32 + lane;
    const uint32_t tbase = tmem_base + ((uint32_t)(quad * 32) << 16);
    uint32_t acc = 0, acc_phase = 0;
    int jq = 0;
    bool ok = true;
    for (int64_t u = u0; ok && u < P.total_units; u += ustep) {
      const VtUnit U = vt_decode<PAIR>(P, u, rank, jq);
      jq = U.job;
      const VtJob& J = P.job[U.job];
      const int m1t = U.m / J.nm2;
      const int m1 = m1t * J.TA + row / J.TB, m2 = (U.m - m1t * J.nm2) * J.TB + row % J.TB;
      const bool valid = m1 < J.M1 && m2 < J.M2;
      const int ncol = J.NT >> 1, c_lo = half * ncol;
      // the unit's sum is kept relative to 2^eref, the largest scale of the
      // job's segments: every block's weight 2^(e - eref) <= 1 is exact in FP32
      int eref = -100000;
      for (int q = lane; q < J.nseg; q += 32) eref = max(eref, seg_exp[J.seg0 + q]);
      eref = __reduce_max_sync(0xffffffffu, eref);
      f2 hi[COLS / 2], lo[COLS / 2];
#pragma unroll
      for (int q = 0; q < COLS / 2; ++q) hi[q] = lo[q] = f2{0ull};
      VtBlock B = vt_first(P, J, U.b_begin);
      for (int64_t b = U.b_begin; b < U.b_end; ++b) {
        const float wk1 = ldexpf(P.seg[B.seg].sign < 0 ? -1.f : 1.f, seg_exp[B.seg] - eref);
        const f2 wk = f2_make(wk1, wk1);
        int got = 0;
        if (!*abort_flag) got = ptx::mbar_wait(&tfull[acc], acc_phase, P.wait_ns) ? 1 : 0;
        // warp-uniform: tcgen05.ld below is .sync.aligned
        if (!__all_sync(0xffffffffu, got)) {
          if (!*abort_flag && lane == 0) vt_abort(P, abort_flag, 24);
          ok = false;
          break;
        }
        ptx::tc_fence_after();
#pragma unroll
        for (int q = 0; q < COLS / LD; ++q) {
          if (LD * q < ncol) {
            const uint32_t cc = acc * 3u * (uint32_t)P.nt_max + (uint32_t)(c_lo + LD * q);
            float a0[LD], a1[LD], a2[LD];
            if constexpr (LD == 8)
              ptx::tmem_ld8x3(tbase + cc, tbase + (uint32_t)J.NT + cc, tbase + 2u * (uint32_t)J.NT + cc, a0, a1, a2);
            else
              ptx::tmem_ld16x3(tbase + cc, tbase + (uint32_t)J.NT + cc, tbase + 2u * (uint32_t)J.NT + cc, a0, a1, a2);
#pragma unroll
            for (int j = 0; j < LD / 2; ++j)
              join<SUM>(hi[LD / 2 * q + j], lo[LD / 2 * q + j], f2_make(a0[2 * j], a0[2 * j + 1]),
                        f2_make(a1[2 * j], a1[2 * j + 1]), f2_make(a2[2 * j], a2[2 * j + 1]), wk);
          }
        }
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (PAIR) ptx::mbar_arrive_cluster(ptx::mapa(&tempty[acc], 0));
          else ptx::mbar_arrive(&tempty[acc]);
        }
        if (++acc == SETS) {
          acc = 0;
          acc_phase ^= 1u;
        }
        vt_next(P, J, B);
      }
      if (!ok || !valid) continue;
      if constexpr (SUM == VT_PAIR) {
        float2* dst = static_cast<float2*>(J.C) + (int64_t)m1 * J.c_m1 + (int64_t)m2 * J.c_m2 + U.n0 + c_lo;
#pragma unroll
        for (int q = 0; q < COLS / 4; ++q) {
          if (4 * q < ncol && U.n0 + c_lo + 4 * q < J.N) {
            float h[4], l[4];
#pragma unroll
            for (int j = 0; j < 2; ++j) {  // the low word can be the larger one
              f2 H, L;
              f2_two_sum(hi[2 * q + j], lo[2 * q + j], H, L);
              f2_get(H, h[2 * j], h[2 * j + 1]);
              f2_get(L, l[2 * j], l[2 * j + 1]);
            }
            if (J.vec) {
              asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(dst + 4 * q), "f"(h[0]), "f"(l[0]),
                           "f"(h[1]), "f"(l[1]), "f"(h[2]), "f"(l[2]), "f"(h[3]), "f"(l[3])
                           : "memory");
            } else {
#pragma unroll
              for (int j = 0; j < 4; ++j)
                if (U.n0 + c_lo + 4 * q + j < J.N) dst[4 * q + j] = make_float2(h[j], l[j]);
            }
          }
        }
        continue;
      }
      const double scale = ldexp(1.0, eref);
      double* dst;
      int64_t dn;
      const bool store = J.nsplit > 1 || J.out == VT_STORE;
      if (J.nsplit > 1) {
        dst = J.part + ((int64_t)U.split * ((int64_t)J.M1 * J.M2) + (int64_t)m1 * J.M2 + m2) * J.N;
        dn = 1;
      } else {
        dst = static_cast<double*>(J.C) + (int64_t)m1 * J.c_m1 + (int64_t)m2 * J.c_m2;
        dn = J.c_n;
      }
      dst += (int64_t)(U.n0 + c_lo) * dn;
#pragma unroll
      for (int q = 0; q < COLS / 4; ++q) {
        const int left = J.N - (U.n0 + c_lo + 4 * q);
        if (4 * q < ncol && left > 0) {
          double* d = dst + 4 * q * dn;
          double old[4], x[4];
          bool other = false;
          if (!store && J.vec) {
            asm volatile("ld.global.v4.f64 {%0,%1,%2,%3}, [%4];"
                         : "=d"(old[0]), "=d"(old[1]), "=d"(old[2]), "=d"(old[3])
                         : "l"(d)
                         : "memory");
          } else if (!store) {
#pragma unroll
            for (int j = 0; j < 4; ++j) old[j] = j < left ? d[j * dn] : 0.0;
          }
          float h[4], l[4];
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            f2 H = hi[2 * q + j], L = lo[2 * q + j];
            if constexpr (SUM == VT_ADD) {  // its low word is a sum of its own
              H = f2_add(hi[2 * q + j], L);
              L = f2_sub(L, f2_sub(H, hi[2 * q + j]));
            }
            f2_get(H, h[2 * j], h[2 * j + 1]);
            f2_get(L, l[2 * j], l[2 * j + 1]);
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) x[j] = pair_double(h[j], l[j], eref, &other);
          if (other) {
#pragma unroll
            for (int j = 0; j < 4; ++j) x[j] = pair_convert(h[j], l[j], scale);
          }
          if (!store) {
#pragma unroll
            for (int j = 0; j < 4; ++j) x[j] += old[j];
          }
          if (J.vec) {
            asm volatile("st.global.v4.f64 [%0], {%1,%2,%3,%4};" ::"l"(d), "d"(x[0]), "d"(x[1]), "d"(x[2]),
                         "d"(x[3])
                         : "memory");
          } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (j < left) d[j * dn] = x[j];
          }
        }
      }
    }
  }

  __syncwarp();
  ptx::tc_fence_before();
  __syncthreads();
  if (PAIR) ptx::cluster_sync();  // neither CTA leaves while the other's MMAs or signals may reach it
  if (warp == 1) {
    ptx::tc_fence_after();
    if (PAIR) ptx::tmem_dealloc_pair(tmem_base, P.tmem_cols);
    else ptx::tmem_dealloc(tmem_base, P.tmem_cols);
  }
}

template <int NS>
__global__ void __launch_bounds__(VT_THREADS, 1)
    k_view_tc(const __grid_constant__ VtMaps maps, const __grid_constant__ VtParams P) {
  view_tc_body<NS, false, VT_ADD>(maps, P);
}
template <int NS, int SUM>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(VT_THREADS, 1)
    k_view_tc_pair(const __grid_constant__ VtMaps maps, const __grid_constant__ VtParams P) {
  view_tc_body<NS, true, SUM>(maps, P);
}

__global__ void __launch_bounds__(256) k_vt_reduce(const __grid_constant__ VtParams P) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < P.total_red;
       e += (int64_t)gridDim.x * blockDim.x) {
    int j = 0;
    while (P.job[j].nsplit <= 1 || e >= P.job[j].red0 + (int64_t)P.job[j].M1 * P.job[j].M2 * P.job[j].N) ++j;
    const VtJob& J = P.job[j];
    const int64_t total = (int64_t)J.M1 * J.M2 * J.N, x = e - J.red0;
    double s = 0.0;
#pragma unroll 8
    for (int z = 0; z < J.nsplit; ++z) s += J.part[z * total + x];
    const int64_t m = x / J.N;
    const int n = (int)(x - m * J.N);
    double* cp = static_cast<double*>(J.C) + (m / J.M2) * J.c_m1 + (m % J.M2) * J.c_m2 + (int64_t)n * J.c_n;
    *cp += s;
  }
}

// dst[p][b][c][r] = src[p][b][r][c] through a 64 x 64 shared tile; pairs of
// BF16 elements move as one 32-bit access when every offset is even (`pairs`)
__global__ void __launch_bounds__(256) k_vt_transpose(const unsigned short* __restrict__ src, int64_t src_ps,
                                                       int64_t src_bs, int64_t src_rs, unsigned short* __restrict__ dst,
                                                       int64_t dst_ps, int64_t dst_bs, int64_t dst_cs, int nb, int R,
                                                       int Cc, int pairs) {
  __shared__ unsigned short tile[64][65];
  const int pb = blockIdx.z, p = pb / nb, b = pb - p * nb;
  const int r0 = blockIdx.y * 64, c0 = blockIdx.x * 64;
  const unsigned short* s = src + p * src_ps + b * src_bs;
  unsigned short* d = dst + p * dst_ps + b * dst_bs;
  const int tx = threadIdx.x, ty = threadIdx.y;
  for (int i = ty; i < 64; i += 8) {
    const int r = r0 + i, c = c0 + 2 * tx;
    if (r >= R) continue;
    const unsigned short* sr = s + r * src_rs;
    if (pairs && c + 1 < Cc) {
      const unsigned int w = *reinterpret_cast<const unsigned int*>(sr + c);
      tile[i][2 * tx] = (unsigned short)(w & 0xffffu);
      tile[i][2 * tx + 1] = (unsigned short)(w >> 16);
    } else {
      if (c < Cc) tile[i][2 * tx] = sr[c];
      if (c + 1 < Cc) tile[i][2 * tx + 1] = sr[c + 1];
    }
  }
  __syncthreads();
  for (int i = ty; i < 64; i += 8) {
    const int c = c0 + i, r = r0 + 2 * tx;
    if (c >= Cc) continue;
    unsigned short* dc = d + c * dst_cs;
    if (pairs && r + 1 < R) {
      *reinterpret_cast<unsigned int*>(dc + r) = (unsigned int)tile[2 * tx][i] | ((unsigned int)tile[2 * tx + 1][i] << 16);
    } else {
      if (r < R) dc[r] = tile[2 * tx][i];
      if (r + 1 < R) dc[r + 1] = tile[2 * tx + 1][i];
    }
  }
}

PFN_cuTensorMapEncodeTiled_v12000 vt_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (fn) return fn;
  void* p = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
      q != cudaDriverEntryPointSuccess || !p) {
    cudaGetLastError();
    return nullptr;
  }
  fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  return fn;
}

}  // namespace

void vt_begin(VtBuild* b, int ns, bool pair) {
  // the tables' entries are written whole when they are taken
  b->P.njobs = b->P.nsegs = 0;
  b->P.ns = ns;
  b->nmaps = 0;
  b->pair = pair;
  b->full = false;
  for (int q = 0; q < VT_BANK_MAX; ++q) b->slot[q] = -1;
}

te_status vt_bank_add(VtBank* k, const VtView& v, int rows_r2, int rows_r1, int* idx) {
  if (k->n >= VT_BANK_MAX) return fail(TE_EINVAL, "view GEMM: more than %d tensor maps", VT_BANK_MAX);
  const VtRoles& R = v.roles;
  if (R.k2 != 0 || v.stride[0] != 1 || R.r2 <= 0 || R.s < R.r2 || R.s < R.r1 || (R.r1 >= 0 && R.r1 < R.r2))
    return fail(TE_EINVAL, "view GEMM: bad view roles");
  if ((reinterpret_cast<uintptr_t>(v.base) & 15) != 0) return fail(TE_EINVAL, "view GEMM: base not 16-byte aligned");
  if (rows_r2 < 1 || rows_r2 > 256 || rows_r1 < 1 || rows_r1 > 256) return fail(TE_EINVAL, "view GEMM: box rows");
  PFN_cuTensorMapEncodeTiled_v12000 enc = vt_encoder();
  if (!enc) return fail(TE_ECUDA, "cuTensorMapEncodeTiled entry point not available");
  cuuint64_t gd[5], gs[4];
  cuuint32_t box[5], e1[5];
  uint64_t smax = 16;
  for (int d = 1; d < 5; ++d)
    if (v.dims[d] > 1) smax = std::max<uint64_t>(smax, v.stride[d] * 2);
  for (int d = 0; d < 5; ++d) {
    gd[d] = std::max<uint64_t>(1, v.dims[d]);
    box[d] = 1;
    e1[d] = 1;
    if (d >= 1) {
      const uint64_t sb = v.dims[d] > 1 ? v.stride[d] * 2 : smax;
      if (sb % 16 != 0 || sb >= (1ull << 40)) return fail(TE_EINVAL, "view GEMM: stride of dimension %d", d);
      gs[d - 1] = sb;
    }
  }
  box[R.k2] = VT_KC;
  box[R.r2] = (cuuint32_t)rows_r2;
  if (R.r1 >= 0) box[R.r1] = (cuuint32_t)rows_r1;
  box[R.s] = (cuuint32_t)v.dims[R.s];  // every slice in one copy
  CUtensorMap* m = &k->m[k->n];
  CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(v.base), gd, gs, box, e1,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(TE_ECUDA, "view GEMM: tensor map encoding failed (CUresult %d)", (int)r);
  k->r[k->n] = R;
  k->r[k->n].rows = (int16_t)(rows_r2 * rows_r1);
  *idx = k->n++;
  return TE_OK;
}

int vt_use(VtBuild* b, const VtBank& k, int idx) {
  if (idx < 0 || idx >= k.n) return -1;
  if (b->slot[idx] >= 0) return b->slot[idx];
  if (b->nmaps >= VT_MAX_MAPS) return -1;
  b->maps.m[b->nmaps] = k.m[idx];
  b->P.roles[b->nmaps] = k.r[idx];
  b->slot[idx] = (int8_t)b->nmaps;
  return b->nmaps++;
}

int64_t vt_seg_blocks(int K1, int K2, int bchunks) {
  const int64_t nchunks = (int64_t)K1 * ((K2 + VT_KC - 1) / VT_KC);
  return (nchunks + bchunks - 1) / bchunks;
}

VtJob* vt_job(VtBuild* b, int M1, int M2, int N, int TA, int TB, int NT, void* C, int64_t c_m1, int64_t c_m2,
              int64_t c_n, VtOut out) {
  if (b->P.njobs >= VT_MAX_JOBS) {
    b->full = true;
    return nullptr;
  }
  VtJob* j = &b->P.job[b->P.njobs++];
  *j = VtJob{};
  j->M1 = M1;
  j->M2 = M2;
  j->N = N;
  j->TA = (int16_t)TA;
  j->TB = (int16_t)TB;
  j->NT = (int16_t)NT;
  j->nm2 = (M2 + TB - 1) / TB;
  const int nm = (M1 + TA - 1) / TA * j->nm2;
  j->nmu = b->pair ? (nm + 1) / 2 : nm;
  j->nn = (N + NT - 1) / NT;
  j->nsplit = 1;
  j->seg0 = (int16_t)b->P.nsegs;
  j->bchunks = VT_BLOCK_CHUNKS;
  j->C = C;
  j->c_m1 = c_m1;
  j->c_m2 = c_m2;
  j->c_n = c_n;
  j->out = (int16_t)out;
  return j;
}

void vt_seg(VtBuild* b, int amap, int bmap, int K1, int K2, const int* afix, const int* bfix, const int* ea,
            const int* eb, int sign) {
  if (b->P.nsegs >= VT_MAX_SEGS || b->P.njobs == 0 || amap < 0 || bmap < 0) {  // vt_finish reports it
    b->full = true;
    return;
  }
  VtJob& j = b->P.job[b->P.njobs - 1];
  ++j.nseg;
  VtSeg& s = b->P.seg[b->P.nsegs++];
  s.amap = (int8_t)amap;
  s.bmap = (int8_t)bmap;
  s.nk2c = (K2 + VT_KC - 1) / VT_KC;
  s.nchunks = K1 * s.nk2c;
  for (int d = 0; d < 3; ++d) {
    s.afix[d] = (int16_t)(afix ? afix[d] : 0);
    s.bfix[d] = (int16_t)(bfix ? bfix[d] : 0);
  }
  s.ea = ea;
  s.eb = eb;
  s.sign = (int16_t)sign;
  j.nblocks += (s.nchunks + VT_BLOCK_CHUNKS - 1) / VT_BLOCK_CHUNKS;
}

int64_t vt_splits(int64_t tiles, int64_t nblocks, int units_at_once) {
  // jobs with long K only (the partials cost a reduction pass): enough units
  // for about four waves over the SMs, and at most 64 blocks per unit
  if (nblocks < 8) return 1;
  const int64_t want = std::max<int64_t>((nblocks + 63) / 64, (4LL * units_at_once + tiles - 1) / tiles);
  return std::max<int64_t>(1, std::min<int64_t>(nblocks, want));
}

te_status vt_finish(VtBuild* b, int num_sms, double* part_scratch, int64_t scratch_cap, int64_t* used) {
  if (b->full) return fail(TE_EINVAL, "view GEMM: launch tables full, or a segment without a tensor map");
  const int at_once = std::max(1, b->pair ? num_sms / 2 : num_sms);
  int64_t units = 0, off = 0, red = 0, launch_tiles = 0;
  for (int q = 0; q < b->P.njobs; ++q) launch_tiles += (int64_t)b->P.job[q].nmu * b->P.job[q].nn;
  for (int q = 0; q < b->P.njobs; ++q) {
    VtJob& J = b->P.job[q];
    if (J.nseg == 0) return fail(TE_EINVAL, "view GEMM: job without segments");
    if (J.out != b->P.job[0].out || (J.out == VT_PAIR && !b->pair))
      return fail(TE_EINVAL, "view GEMM: one output kind per launch; VT_PAIR on CTA pairs");
    int kblocks = 0;
    for (int g = J.seg0; g < J.seg0 + J.nseg; ++g) {
      const VtSeg& S = b->P.seg[g];
      if (S.sign != 1 && S.sign != -1) return fail(TE_EINVAL, "view GEMM: segment factor other than +-1");
      if (b->P.roles[S.amap].rows != 128 || b->P.roles[S.bmap].rows != (b->pair ? J.NT / 2 : J.NT))
        return fail(TE_EINVAL, "view GEMM: box rows do not fit the tile");
      kblocks += (S.nchunks + VT_SPLIT_CHUNKS - 1) / VT_SPLIT_CHUNKS;
    }
    // the other jobs of the launch share the SMs: a job alone gets its part of them
    const int64_t tiles = (int64_t)J.nmu * J.nn;
    const int64_t share = std::max<int64_t>(1, at_once * tiles / std::max<int64_t>(1, launch_tiles));
    int64_t ns = 1;
    if (J.out == VT_ADD && part_scratch && launch_tiles < at_once && J.nblocks * VT_BLOCK_CHUNKS >= 8 * VT_SPLIT_CHUNKS) {
      J.bchunks = VT_SPLIT_CHUNKS;
      J.nblocks = kblocks;
    }
    if (J.out == VT_ADD && part_scratch) ns = vt_splits(tiles, J.nblocks, (int)share);
    const int64_t mn = (int64_t)J.M1 * J.M2 * J.N;
    while (ns > 1 && off + ns * mn > scratch_cap) ns = std::max<int64_t>(1, ns / 2);
    J.nsplit = (int)ns;
    J.part = nullptr;
    J.red0 = 0;
    if (ns > 1) {
      J.part = part_scratch + off;
      off += (ns * mn + 3) / 4 * 4;
      J.red0 = red;
      red += mn;
    }
    // four columns per access: contiguous, whole groups of four, 32-byte aligned
    const int64_t es = 8;
    if (ns > 1) J.vec = J.N % 4 == 0 ? 1 : 0;
    else
      J.vec = J.c_n == 1 && J.N % 4 == 0 && J.c_m1 % 4 == 0 && J.c_m2 % 4 == 0 &&
              (reinterpret_cast<uintptr_t>(J.C) % (4 * es)) == 0;
    if (ns > 1 && (reinterpret_cast<uintptr_t>(J.part) % (4 * es)) != 0) J.vec = 0;
    J.unit0 = units;
    units += tiles * ns;
  }
  b->P.total_units = units;
  b->P.total_red = red;
  if (used) *used = off;
  return TE_OK;
}

int64_t vt_split_doubles(int64_t tiles, int64_t nblocks, int64_t mn, int units_at_once) {
  const int64_t ns = vt_splits(tiles, nblocks, units_at_once);
  return ns > 1 ? ns * mn : 0;
}

template <int NS>
static cudaError_t vt_launch_ns(const VtBuild* b, int grid, size_t smem, cudaStream_t s) {
  auto* k = k_view_tc<NS>;
  if (b->pair) {
    const int out = b->P.job[0].out;
    k = out == VT_STORE ? k_view_tc_pair<NS, VT_STORE> : (out == VT_PAIR ? k_view_tc_pair<NS, VT_PAIR> : k_view_tc_pair<NS, VT_ADD>);
  }
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k<<<(unsigned)grid, VT_THREADS, smem, s>>>(b->maps, b->P);
  return cudaGetLastError();
}

te_status vt_launch(Handle* h, VtBuild* b, cudaStream_t s) {
  VtParams& P = b->P;
  if (P.total_units == 0) return TE_OK;
  int nt_max = 16;
  for (int q = 0; q < P.njobs; ++q) {
    const VtJob& J = P.job[q];
    if (J.NT % (b->pair ? 32 : 16) != 0 || J.NT < 16 || J.NT > (b->pair ? VT_NT_PAIR : VT_NT_MAX) || J.TA * J.TB != 128)
      return fail(TE_EINVAL, "view GEMM: tile %d x %d x %d", J.TA, J.TB, J.NT);
    nt_max = std::max<int>(nt_max, J.NT);
  }
  P.nt_max = nt_max;
  P.stage_bytes = (uint32_t)P.ns * (VT_A_SLICE + (uint32_t)(b->pair ? nt_max / 2 : nt_max) * VT_ROW_BYTES);
  const size_t avail = h->smem_optin > 4096 ? h->smem_optin - 4096 : 0;
  P.stages = (int)std::min<size_t>(8, avail / P.stage_bytes);
  if (P.stages < 2) return fail(TE_EUNSUPPORTED, "view GEMM: not enough shared memory for two stages");
  uint32_t cols = 32;
  while (cols < (b->pair ? 6u : 3u) * (uint32_t)nt_max) cols <<= 1;
  P.tmem_cols = cols;
  P.err = h->d_err;
  P.wait_ns = h->wait_limit_ns;
  const size_t smem = (size_t)P.stages * P.stage_bytes + 1024 + 256;
  const int grid = b->pair ? 2 * (int)std::min<int64_t>(P.total_units, std::max(1, h->num_sms / 2))
                           : (int)std::min<int64_t>(P.total_units, std::max(1, h->num_sms));
  cudaError_t e = P.ns == 5 ? vt_launch_ns<5>(b, grid, smem, s) : vt_launch_ns<4>(b, grid, smem, s);
  if (e != cudaSuccess) return fail(TE_ECUDA, "view GEMM launch: %s", cudaGetErrorString(e));
  ++h->n_launches;
  if (P.total_red > 0) {
    k_vt_reduce<<<(unsigned)std::min<int64_t>((P.total_red + 255) / 256, 4 * std::max(1, h->num_sms)), 256, 0, s>>>(P);
    ++h->n_launches;
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) return fail(TE_ECUDA, "view GEMM reduce: %s", cudaGetErrorString(e));
  return TE_OK;
}

int vt_ntile(int64_t n, bool pair) {
  // cta_group::2 takes N in steps of 32.  Lone CTAs in steps of 16 do less for padding:
  // nvir = 320 in 3 x 112 columns 2.50 ms per triple, in 3 x 128 2.64
  const int64_t most = pair ? VT_NT_PAIR : VT_NT_MAX, step = pair ? 32 : 16, t = (n + most - 1) / most;
  return (int)(((n + t - 1) / t + step - 1) / step * step);
}

te_status vt_product(Handle* h, const void* a, int64_t a_plane, int64_t m, const void* b, int64_t b_plane, int64_t n,
                     int64_t K, int64_t Kp, int ns, const int* ea, const int* eb, double* C, cudaStream_t s) {
  const VtRoles ROW{0, 1, -1, -1, 2, 0};
  const int NT = vt_ntile(n, false);
  VtBank bank;
  bank.n = 0;
  int ma = 0, mb = 0;
  const uint64_t NS = (uint64_t)ns;
  const VtView va{a, {(uint64_t)K, (uint64_t)m, NS, 1, 1}, {1, (uint64_t)Kp, (uint64_t)a_plane, 0, 0}, ROW};
  const VtView vb{b, {(uint64_t)K, (uint64_t)n, NS, 1, 1}, {1, (uint64_t)Kp, (uint64_t)b_plane, 0, 0}, ROW};
  te_status st = vt_bank_add(&bank, va, 128, 1, &ma);
  if (st == TE_OK) st = vt_bank_add(&bank, vb, NT, 1, &mb);
  if (st != TE_OK) return st;
  std::unique_ptr<VtBuild> B(new (std::nothrow) VtBuild);
  if (!B) return fail(TE_ENOMEM, "view GEMM tables");
  vt_begin(B.get(), ns, false);
  const int none[3] = {0, 0, 0};
  VtJob* j = vt_job(B.get(), 1, (int)m, (int)n, 1, 128, NT, C, 0, n, 1, VT_STORE);
  vt_seg(B.get(), vt_use(B.get(), bank, ma), vt_use(B.get(), bank, mb), 1, (int)K, none, none, ea, eb, 1);
  j->bchunks = VT_PRODUCT_CHUNKS;
  j->nblocks = vt_seg_blocks(1, (int)K, VT_PRODUCT_CHUNKS);
  st = vt_finish(B.get(), h->num_sms, nullptr, 0, nullptr);
  return st == TE_OK ? vt_launch(h, B.get(), s) : st;
}

te_status vt_slice_maps(VtBank* k, const SliceSet& S, int o, int v, int nt, int* idx) {
  const uint64_t V = (uint64_t)v, O = (uint64_t)o, NS = (uint64_t)S.ns, vp = (uint64_t)S.vp, op = (uint64_t)S.op;
  const VtRoles XY{0, 1, 2, -1, 3}, ROW{0, 1, -1, -1, 2};
  struct Spec {
    const void* base;
    uint64_t dims[5], str[5];
    VtRoles r;
    int rows2, rows1;
  } sp[6] = {
      {S.ovvv, {V, V, V, NS, O}, {1, vp, V * vp, (uint64_t)S.ovvv_plane, (uint64_t)S.ovvv_p}, XY, 16, 8},
      {S.ovvv, {V, V, V, NS, O}, {1, V * vp, vp, (uint64_t)S.ovvv_plane, (uint64_t)S.ovvv_p}, XY, 16, 8},
      {S.t2L, {O, V, V, NS, O}, {1, op, V * op, (uint64_t)S.t2L_plane, (uint64_t)S.t2L_q}, XY, 16, 8},
      {S.t2L, {O, V, V, NS, O}, {1, V * op, op, (uint64_t)S.t2L_plane, (uint64_t)S.t2L_q}, XY, 16, 8},
      {S.t2, {V, V, NS, O, O}, {1, vp, (uint64_t)S.t2_plane, (uint64_t)S.t2_rq, O * (uint64_t)S.t2_rq}, ROW, nt / 2, 1},
      {S.nooT, {O, V, NS, O, O}, {1, op, (uint64_t)S.nooT_plane, (uint64_t)S.nooT_pr, O * (uint64_t)S.nooT_pr}, ROW,
       nt / 2, 1},
  };
  for (int q = 0; q < 6; ++q) {
    VtView w;
    w.base = sp[q].base;
    for (int d = 0; d < 5; ++d) {
      w.dims[d] = sp[q].dims[d];
      w.stride[d] = sp[q].str[d];
    }
    w.roles = sp[q].r;
    const te_status st = vt_bank_add(k, w, sp[q].rows2, sp[q].rows1, &idx[q]);
    if (st != TE_OK) return st;
  }
  return TE_OK;
}

cudaError_t vt_transpose(const void* src, int64_t src_ps, int64_t src_bs, int64_t src_rs, void* dst, int64_t dst_ps,
                         int64_t dst_bs, int64_t dst_cs, int np, int nb, int R, int Cc, cudaStream_t s) {
  if (np <= 0 || nb <= 0 || R <= 0 || Cc <= 0 || (R + 63) / 64 > 65535) return cudaErrorInvalidValue;
  const int pairs = (((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 3) == 0 &&
                     ((src_ps | src_bs | src_rs | dst_ps | dst_bs | dst_cs) & 1) == 0)
                        ? 1
                        : 0;
  const unsigned short* s16 = static_cast<const unsigned short*>(src);
  unsigned short* d16 = static_cast<unsigned short*>(dst);
  // the grid's z extent covers (plane, batch) pairs: planes in groups when
  // all batches fit, else one plane at a time in batch chunks
  if (nb <= 65535) {
    const int per = std::max(1, std::min(np, 65535 / nb));
    for (int p0 = 0; p0 < np; p0 += per) {
      const int n = std::min(per, np - p0);
      dim3 grid((unsigned)((Cc + 63) / 64), (unsigned)((R + 63) / 64), (unsigned)(n * nb));
      k_vt_transpose<<<grid, dim3(32, 8), 0, s>>>(s16 + p0 * src_ps, src_ps, src_bs, src_rs, d16 + p0 * dst_ps, dst_ps,
                                                   dst_bs, dst_cs, nb, R, Cc, pairs);
    }
  } else {
    for (int p0 = 0; p0 < np; ++p0)
      for (int b0 = 0; b0 < nb; b0 += 65535) {
        const int n = std::min(65535, nb - b0);
        dim3 grid((unsigned)((Cc + 63) / 64), (unsigned)((R + 63) / 64), (unsigned)n);
        k_vt_transpose<<<grid, dim3(32, 8), 0, s>>>(s16 + p0 * src_ps + b0 * src_bs, src_ps, src_bs, src_rs,
                                                     d16 + p0 * dst_ps + b0 * dst_bs, dst_ps, dst_bs, dst_cs, n, R, Cc,
                                                     pairs);
      }
  }
  return cudaGetLastError();
}

}  // namespace te
