// Tensor-core path (TF32, BF16x3, TF32x3, OZAKI) for the W~ contractions.
//
// The same three G blocks as the float64 path (see gemm_fp64.cu):
//   W~_{ijk}[a,b,c] = G(i,j,k)[a,b,c] + G(j,k,i)[b,c,a] + G(k,i,j)[c,a,b]
// each one GEMM  D[(x,y), z] = sum_K A[(x,y), K] B[z, K]  with four K segments
//   S1 ovvv[p,x,y,:] . t2[r,q,z,:]     S2 ovvv[q,y,x,:] . t2[r,p,z,:]
//   S3 t2L[p,y,x,:] . nooT[q,r,z,:]    S4 t2L[q,x,y,:] . nooT[p,r,z,:]
// run on tcgen05 by pairs of CTAs (cta_group::2, the two SMs of a TPC): a pair
// takes two 128-row A tiles (TA values of x times TB of y each) against one
// B tile of NT rows, of which each CTA holds half.  TMA brings each CTA's part
// into its swizzled shared memory; one thread of the pair's first CTA issues
// the MMAs for both SMs into FP32 accumulators in tensor memory; eight epilogue
// warps per CTA drain its TMEM into the G buffer.
//
// Why pairs, and who issues.  The ten slice products of a K step read their
// operands from shared memory again each time; in a pair each SM reads its own
// 128 A rows but only NT / 2 B rows, loads half of B, and four pipeline stages
// fit instead of three.  That pays only once the issue keeps up: issued from a
// single-thread branch, an MMA took 75 to 80 cycles whatever its N, because its
// operands went to uniform registers one by one (see the issuer).  Main loop
// plus stores of four triples at nvir = 320 (and the whole nocc=24 nvir=240
// contraction): 3.10 ms (956 ms) lone CTAs and a single issuing thread; 3.10 ms
// (931 ms) pairs alone; 3.15 ms (856 ms) uniform issue alone; 2.78 ms (711 ms)
// both, 1.99 PFLOP/s of slice products at nvir = 320.  Tried on top and not
// kept: a second place for the third accumulator where NT <= 128 leaves TMEM
// for it (2% slower), sixteen epilogue warps (7% slower: spills), 128-byte
// operand rows in two stages (7% slower).
//
// Operand forms, prepared once per call:
//  * TF32, BF16X3, TF32X3: x = hi + lo, hi and lo the nearest 11-bit (TF32)
//    or 8-bit (BF16) significands (Veltkamp splitting); the products
//    hi*hi + hi*lo + lo*hi (hi*hi only for TF32) share one accumulator.
//  * OZAKI (Ozaki, Ogita, Oishi, Rump 2012, error-free slicing): each array
//    is scaled by 2^-s (s from its largest magnitude, chosen so that every
//    segment of the K axis has the same unit) and cut into four slices
//    m_k 2^-7k, |m_k| <= 128, exact in BF16.  Slice products are then exact
//    multiples of 2^-7(k+l); the level-2 product and the two level-3
//    products each go to their own accumulator, where every partial sum is
//    an integer multiple of the level's unit below 2^24 units - exact, so the
//    tensor core's FP32 accumulation cannot round them.  The seven products
//    of levels 4 and 5 share a third accumulator.  The epilogue adds the
//    three with an exact two-sum and stores G as an FP32 pair (hi, lo).
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdio>
#include <cstring>

#include "energy_tc.h"
#include "prep_tc.h"
#include "ptx_sm100.cuh"
#include "strided.h"
#include "tc_path.h"
#include "view_tc.h"

namespace te {

constexpr int OZ_K_MAX7 = 1024;  // K * 2^14 < 2^24: exact level-2/3 sums with 7-bit slices
constexpr int OZ_K_MAX6 = 4096;  // K * 2^12 < 2^24 with 6-bit slices

// ozaki_bits: 0 = 7-bit slices when K allows, else 6-bit; 6 or 7 forces one.
static int tc_mode_of(te_precision p, int o, int v, int ozaki_bits) {
  switch (p) {
    case TE_TF32: return TC_TF32;
    case TE_BF16X3: return TC_BF16X3;
    case TE_TF32X3: return TC_TF32X3;
    default:
      if (ozaki_bits == 6) return TC_OZAKI6;
      if (ozaki_bits == 7) return TC_OZAKI;
      return 2 * (v + o) <= OZ_K_MAX7 ? TC_OZAKI : TC_OZAKI6;
  }
}

// ---------------------------------------------------------------------------
// the GEMM kernel
// ---------------------------------------------------------------------------

// One 5-D map per operand view; the slice is a box dimension, so one copy
// brings every slice of a stage (the slices land part-contiguous in shared
// memory, as the MMA descriptors expect).
struct TcMaps {
  CUtensorMap a_nat;  // ovvv slices [p][s][x][y][Kp], dims (Kp, y, x, s, p): rows (x,y) of ovvv[p]
  CUtensorMap a_tr;   // the same with the y and x strides swapped: rows ovvv[q,y,x,:]
  CUtensorMap l_nat;  // t2L slices [q][s][x][y][op], natural
  CUtensorMap l_tr;   // t2L slices, transposed rows
  CUtensorMap b_t2;   // t2 slices [r][q][s][z][Kp], dims (Kp, z, s, q, r)
  CUtensorMap b_noo;  // nooT slices [p][r][s][z][op], dims (op, z, s, r, p)
};

// The maps of every cluster of a launch.
struct TcMapSet {
  TcMaps m[TC_MAX_CL];
};

// Per-cluster constants of a contraction launch.
struct TcCl {
  int o, v;
  int TA, TB, NT;
  int n_my, n_mp, n_nt;    // M tiles along y; pairs of M tiles; N tiles
  int kw_chunks, ko_chunks;
  int kw_elems, ko_elems;  // elements per chunk
  int cbo;                 // chunk bytes of the o-segments (the v-segments use TcParams::cbw)
  int64_t slot_floats;     // G floats per triple slot
  const int* exps;         // OZAKI scale exponents
};

struct TcParams {
  int ncl, npieces;
  int cbw;                 // chunk bytes of the v-segments
  int stages;
  uint32_t stage_bytes;    // stage stride: the largest cluster's A and B parts
  uint32_t a_part_bytes;   // 128 rows x cbw
  uint32_t tmem_cols;
  int nbuf;                // TMEM accumulator sets (1 or 2)
  int fmt;                 // G format
  int nt_max;              // largest N tile: stride of the accumulator sets
  int64_t total_tiles;     // pair tiles
  const Triple* triples;
  unsigned int* err;
  unsigned long long wait_ns;
  TcCl cl[TC_MAX_CL];
  TcPiece pc[TC_MAX_PIECES];
};

__device__ __forceinline__ uint32_t layout_code(int cb) { return cb == 128 ? 2u : (cb == 64 ? 4u : 6u); }

__device__ __forceinline__ void record_abort(const TcParams& P, volatile int* abort_flag, unsigned site) {
  *abort_flag = 1;
  if (atomicOr(P.err, ERR_WAIT_TIMEOUT) == 0) {
    P.err[1] = site;
    P.err[2] = blockIdx.x;
  }
}

struct TileCoord {
  int cl, piece, slot, g, p, q, r, x0, y0, z0;
};

// the cluster of tile tt
__device__ __forceinline__ int tile_cluster(const TcParams& P, int64_t tt) {
  int q = 0;  // pieces are in tile order
  while (q + 1 < P.npieces && P.pc[q + 1].tile0 <= tt) ++q;
  return P.pc[q].cl;
}

// pair tile tt; x0 and y0 are those of CTA `rank`'s M tile (the second tile of an
// odd last pair lies beyond x < v: its loads fill zeros, its rows are not stored)
__device__ __forceinline__ TileCoord decode_tile(const TcParams& P, int64_t tt, int rank) {
  TileCoord c;
  int q = 0;  // pieces are in tile order
  while (q + 1 < P.npieces && P.pc[q + 1].tile0 <= tt) ++q;
  const TcPiece& pc = P.pc[q];
  const TcCl& C = P.cl[pc.cl];
  int64_t rest = tt - pc.tile0;
  const int nt = (int)(rest % C.n_nt);
  rest /= C.n_nt;
  const int m = 2 * (int)(rest % C.n_mp) + rank;
  rest /= C.n_mp;
  const int mx = m / C.n_my, my = m - mx * C.n_my;
  c.g = (int)(rest % 3);
  c.slot = (int)(rest / 3);
  c.cl = pc.cl;
  c.piece = q;
  const Triple T = P.triples[pc.t0 + c.slot];
  if (c.g == 0) { c.p = T.i; c.q = T.j; c.r = T.k; }
  else if (c.g == 1) { c.p = T.j; c.q = T.k; c.r = T.i; }
  else { c.p = T.k; c.q = T.i; c.r = T.j; }
  c.x0 = mx * C.TA;
  c.y0 = my * C.TB;
  c.z0 = nt * C.NT;
  return c;
}

// out[k] = v[k ^ h] for k < 8 (three conditional swap stages, no dynamic indexing)
__device__ __forceinline__ void xor_permute8(float* v, int h) {
  if (h & 1) {
#pragma unroll
    for (int k = 0; k < 8; k += 2) { const float t = v[k]; v[k] = v[k + 1]; v[k + 1] = t; }
  }
  if (h & 2) {
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if ((k & 2) == 0) { const float t = v[k]; v[k] = v[k + 2]; v[k + 2] = t; }
  }
  if (h & 4) {
#pragma unroll
    for (int k = 0; k < 4; ++k) { const float t = v[k]; v[k] = v[k + 4]; v[k + 4] = t; }
  }
}

// the same for eight 16-bit values, two per word
__device__ __forceinline__ uint4 xor_permute8_packed(const uint32_t* v, int h) {
  uint32_t a = v[0], b = v[1], c = v[2], d = v[3], t;
  if (h & 1) {
    a = __byte_perm(a, 0, 0x1032);
    b = __byte_perm(b, 0, 0x1032);
    c = __byte_perm(c, 0, 0x1032);
    d = __byte_perm(d, 0, 0x1032);
  }
  if (h & 2) { t = a; a = b; b = t; t = c; c = d; d = t; }
  if (h & 4) { t = a; a = c; c = t; t = b; b = d; d = t; }
  return make_uint4(a, b, c, d);
}

// one 32-byte sector in one store (dst 32-byte aligned)
__device__ __forceinline__ void store8(float* dst, const float* v) {
  asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(dst), "f"(v[0]), "f"(v[1]), "f"(v[2]),
               "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
               : "memory");
}

// Knuth's two-sum: s + e == a + b exactly
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// Warp roles: 0 TMA producer, 1 MMA issuer (and TMEM owner), the rest
// epilogue: warp w drains TMEM lanes 32 (w % 4) .. +31 (the lane quarter its
// warp index may access) and every (GEMM_EPI_WARPS / 4)-th 16-column chunk,
// starting at chunk (w - 2) / 4.
constexpr int GEMM_EPI_WARPS = 8;
constexpr int GEMM_EPI_GROUPS = GEMM_EPI_WARPS / 4;
constexpr int GEMM_THREADS = (2 + GEMM_EPI_WARPS) * 32;
// 16-column chunks one epilogue warp holds in registers with a single
// accumulator set (exact-slice N tiles of at most 160 columns)
constexpr int EPI_CHUNKS = 5;
constexpr int EPI_NT_MAX = 16 * GEMM_EPI_GROUPS * EPI_CHUNKS;
constexpr int EPI_NT_LO32 = 96;  // the widest such tile whose low words stay FP32
constexpr int GEMM_PAIR = 2;  // CTAs per cluster

// LO32: G's low words are FP32 (G_PAIR), else BF16 where they are held in
// registers (G_MIXED); the exact-slice modes only
template <int MODE, bool LO32>
__global__ void __cluster_dims__(GEMM_PAIR, 1, 1) __launch_bounds__(GEMM_THREADS, 1)
    k_gemm_tc(const __grid_constant__ TcMapSet maps, const __grid_constant__ TcParams P) {
  using MT = ModeTraits<MODE>;
  constexpr bool TF32 = MT::tf32;
  constexpr int NPART = MT::nparts;
  constexpr int NACC = MT::nacc;
  // TMEM accumulator sets: 2 when they fit (the epilogue of one tile then
  // overlaps the MMAs of the next), else 1
  const int NBUF = P.nbuf;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                         ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + (size_t)P.stages * P.stage_bytes);
  uint64_t* empty = full + P.stages;
  uint64_t* tfull = empty + P.stages;
  uint64_t* tempty = tfull + 2;
  uint64_t* drain = tempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int rank = (int)ptx::cluster_ctarank();  // rank 0 issues the pair's MMAs
  const int64_t pair0 = blockIdx.x / GEMM_PAIR, npairs = gridDim.x / GEMM_PAIR;

  if (threadIdx.x == 0) {
    for (int s = 0; s < P.stages; ++s) {
      ptx::mbar_init(&full[s], 1);
      ptx::mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      ptx::mbar_init(&tfull[a], 1);
      ptx::mbar_init(&tempty[a], GEMM_PAIR * GEMM_EPI_WARPS);
    }
    ptx::mbar_init(drain, 1);
    *abort_flag = 0;
    ptx::fence_barrier_init();
  }
  if (warp == 0 && lane < P.ncl) {
    const TcMaps& m = maps.m[lane];
    ptx::tma_prefetch_desc(&m.a_nat);
    ptx::tma_prefetch_desc(&m.a_tr);
    ptx::tma_prefetch_desc(&m.l_nat);
    ptx::tma_prefetch_desc(&m.l_tr);
    ptx::tma_prefetch_desc(&m.b_t2);
    ptx::tma_prefetch_desc(&m.b_noo);
  }
  if (warp == 1) {
    ptx::tmem_alloc_pair(tmem_slot, P.tmem_cols);
    ptx::tmem_relinquish_pair();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::cluster_sync();  // the barriers of both CTAs are initialised before either is signalled
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const uint32_t acc_stride = (uint32_t)(NACC * P.nt_max);  // TMEM columns between accumulator sets

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      uint32_t stage = 0, phase = 0;
      int pending[16];
      for (int s = 0; s < 16; ++s) pending[s] = -1;
      bool ok = true;
      for (int64_t tt = pair0; ok && tt < P.total_tiles; tt += npairs) {
        const TileCoord c = decode_tile(P, tt, rank);
        const TcCl& C = P.cl[c.cl];
        const TcMaps& mp = maps.m[c.cl];
        for (int seg = 0; ok && seg < 4; ++seg) {
          const bool wide = seg < 2;
          const int nch = wide ? C.kw_chunks : C.ko_chunks;
          const int cb = wide ? P.cbw : C.cbo;
          const int ce = wide ? C.kw_elems : C.ko_elems;
          const uint32_t bytes = (uint32_t)NPART * (2u * 128u * cb + (uint32_t)C.NT * cb);  // both CTAs'
          for (int ch = 0; ch < nch; ++ch) {
            if (*abort_flag || !ptx::mbar_wait(&empty[stage], phase ^ 1u, P.wait_ns)) {
              if (!*abort_flag) record_abort(P, abort_flag, 1);
              ok = false;
              break;
            }
            // the pair's bytes all count on rank 0's barrier, whose MMAs wait for them
            if (rank == 0) ptx::mbar_arrive_expect_tx(&full[stage], bytes);
            const uint32_t bar = ptx::mapa(&full[stage], 0);
            pending[stage] = (int)phase;
            unsigned char* sa = smem + (size_t)stage * P.stage_bytes;
            unsigned char* sb = sa + NPART * P.a_part_bytes;
            const int kc = ch * ce, zr = c.z0 + rank * (C.NT / 2);
            if (seg == 0) {
              ptx::tma_load_5d_pair(sa, &mp.a_nat, bar, kc, c.y0, c.x0, 0, c.p);
              ptx::tma_load_5d_pair(sb, &mp.b_t2, bar, kc, zr, 0, c.q, c.r);
            } else if (seg == 1) {
              ptx::tma_load_5d_pair(sa, &mp.a_tr, bar, kc, c.y0, c.x0, 0, c.q);
              ptx::tma_load_5d_pair(sb, &mp.b_t2, bar, kc, zr, 0, c.p, c.r);
            } else if (seg == 2) {
              ptx::tma_load_5d_pair(sa, &mp.l_tr, bar, kc, c.y0, c.x0, 0, c.p);
              ptx::tma_load_5d_pair(sb, &mp.b_noo, bar, kc, zr, 0, c.r, c.q);
            } else {
              ptx::tma_load_5d_pair(sa, &mp.l_nat, bar, kc, c.y0, c.x0, 0, c.q);
              ptx::tma_load_5d_pair(sb, &mp.b_noo, bar, kc, zr, 0, c.r, c.p);
            }
            if (++stage == (uint32_t)P.stages) {
              stage = 0;
              phase ^= 1u;
            }
          }
        }
      }
      // Before the pair exits: the MMAs have released every stage (their
      // signals reach both CTAs), so every copy has landed too.  After an
      // expired wait they may not come: rank 0 waits for the copies it
      // expects, and both for longer than a copy takes.
      for (int s = 0; s < P.stages; ++s) {
        if (pending[s] < 0) continue;
        if (ok && !*abort_flag) ptx::mbar_wait(&empty[s], (uint32_t)pending[s], P.wait_ns);
        else if (rank == 0) ptx::mbar_wait(&full[s], (uint32_t)pending[s], P.wait_ns);
      }
      if (!ok || *abort_flag) ptx::pause_ns(200000);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (rank 0, for both SMs) ----------------
    // The whole warp runs this loop, its branches decided by votes, and one
    // elected lane issues: descriptors and addresses are then warp-uniform
    // values in uniform registers, where tcgen05.mma takes its operands.  In a
    // single-thread branch they were moved there one by one, 75 to 80 cycles
    // per MMA whatever its N (64 cycles of tensor work at N = 128).
    const uint32_t fmt = TF32 ? 2u : 1u;
    uint32_t stage = 0, phase = 0, acc = 0, acc_phase = 0;
    bool ok = true;
    bool issued = false;
    auto wait_all = [&](uint64_t* bar, uint32_t parity, unsigned site) -> bool {
      const int got = (!*abort_flag && ptx::mbar_wait(bar, parity, P.wait_ns)) ? 1 : 0;
      const bool all = __all_sync(0xffffffffu, got);
      if (!all && lane == 0 && !*abort_flag) record_abort(P, abort_flag, site);
      return all;
    };
    const uint32_t smem0 = ptx::smem_u32(smem);
    for (int64_t tt = pair0; ok && rank == 0 && tt < P.total_tiles; tt += npairs) {
      const TcCl& C = P.cl[tile_cluster(P, tt)];
      const uint32_t NT = (uint32_t)C.NT;
      const uint32_t idesc = (1u << 4) | (fmt << 7) | (fmt << 10) | ((NT >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
      if (!wait_all(&tempty[acc], acc_phase ^ 1u, 2)) break;
      ptx::tc_fence_after();
      const uint32_t d_tmem = tmem_base + acc * acc_stride;
      uint32_t first = 1;
      for (int seg = 0; ok && seg < 4; ++seg) {
        const bool wide = seg < 2;
        const int nch = wide ? C.kw_chunks : C.ko_chunks;
        const uint32_t cb = wide ? (uint32_t)P.cbw : (uint32_t)C.cbo;
        // one box per operand lands the slices back to back: 128 (A) or NT / 2 (B) rows of cb bytes each
        const uint64_t desc0 = ptx::smem_desc(0, 8u * cb, layout_code((int)cb));
        const uint32_t astep = (128u * cb) >> 4, bstep = (NT / 2 * cb) >> 4;  // slices, in descriptor units
        for (int ch = 0; ch < nch; ++ch) {
          if (!wait_all(&full[stage], phase, 3)) {
            ok = false;
            break;
          }
          ptx::tc_fence_after();
          const uint32_t a0 = (smem0 + stage * P.stage_bytes) >> 4;
          const uint32_t b0 = a0 + ((NPART * P.a_part_bytes) >> 4);
          for (uint32_t ks = 0; ks < cb / 32; ++ks) {
            uint64_t ad[NPART], bd[NPART];
#pragma unroll
            for (int k = 0; k < NPART; ++k) {
              ad[k] = desc0 + (a0 + k * astep + ks * 2);
              bd[k] = desc0 + (b0 + k * bstep + ks * 2);
            }
            const uint32_t acc_in = first ? 0u : 1u;
            if (ptx::elect_one()) {
              if constexpr (is_ozaki(MODE)) {
                // slice products a_i b_j with i + j <= NPART - 1: level i + j = 0 and
                // level 1 each in an exact accumulator, the higher levels in a third
                const uint32_t d2 = d_tmem, d3 = d_tmem + NT, dr = d_tmem + 2 * NT;
                ptx::mma_pair<false>(d2, ad[0], bd[0], idesc, acc_in);
                ptx::mma_pair<false>(d3, ad[0], bd[1], idesc, acc_in);
                ptx::mma_acc_pair<false>(d3, ad[1], bd[0], idesc);
                ptx::mma_pair<false>(dr, ad[0], bd[2], idesc, acc_in);
#pragma unroll
                for (int lev = 2; lev < NPART; ++lev)
#pragma unroll
                  for (int i = lev == 2 ? 1 : 0; i <= lev; ++i) ptx::mma_acc_pair<false>(dr, ad[i], bd[lev - i], idesc);
              } else {
                ptx::mma_pair<TF32>(d_tmem, ad[0], bd[0], idesc, acc_in);
                if constexpr (NPART == 2) {
                  ptx::mma_acc_pair<TF32>(d_tmem, ad[0], bd[1], idesc);
                  ptx::mma_acc_pair<TF32>(d_tmem, ad[1], bd[0], idesc);
                }
              }
            }
            first = 0;
          }
          issued = true;
          if (ptx::elect_one()) ptx::mma_commit_pair(&empty[stage]);
          if (++stage == (uint32_t)P.stages) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
      if (!ok) break;
      if (ptx::elect_one()) ptx::mma_commit_pair(&tfull[acc]);
      if (NBUF == 2) {
        acc ^= 1u;
        if (acc == 0) acc_phase ^= 1u;
      } else {
        acc_phase ^= 1u;
      }
    }
    // every issued MMA completes before TMEM is released
    if (issued) {
      if (ptx::elect_one()) ptx::mma_commit_pair_own(drain);
      ptx::mbar_wait(drain, 0, P.wait_ns);
    }
    __syncwarp();
  } else {
    // ---------------- epilogue: TMEM -> G buffer ----------------
    const int quad = warp & 3;
    const int chunk0 = (warp - 2) >> 2;  // this warp's first 16-column chunk
    const int row = quad * 32 + lane;
    uint32_t acc = 0, acc_phase = 0;
    for (int64_t tt = pair0; tt < P.total_tiles; tt += npairs) {
      const TileCoord c = decode_tile(P, tt, rank);
      const TcCl& C = P.cl[c.cl];
      const TcPiece& pc = P.pc[c.piece];
      int got = 0;
      if (!*abort_flag) got = ptx::mbar_wait(&tfull[acc], acc_phase, P.wait_ns) ? 1 : 0;
      // the decision is warp-uniform: tcgen05.ld below is a .sync.aligned instruction
      if (!__all_sync(0xffffffffu, got)) {
        if (!*abort_flag && lane == 0) record_abort(P, abort_flag, 4);
        break;
      }
      ptx::tc_fence_after();
      float gscale = 1.f;
      if (is_ozaki(MODE)) gscale = ldexpf(1.f, C.exps[4]);
      const int x = c.x0 + row / C.TB;
      const int y = c.y0 + row % C.TB;
      const bool valid = x < C.v && y < C.v;
      // orbit-major G: [slot][bt][g][pid][cube], swizzled rows (see
      // energy_tc.h); this row is (x, y) = (X*8 + xl, Y*8 + yl)
      const int nb = (C.v + 7) >> 3;
      constexpr int CUBE = g_cube_floats(is_ozaki(MODE) ? G_PAIR : G_F32);  // with two accumulator sets
      float* const gslot = pc.gbuf + (int64_t)c.slot * C.slot_floats;
      const int roff = cube_row(x & 7, y & 7);
      const int zx = cube_zx(x & 7, y & 7);
      const uint32_t tbase = tmem_base + ((uint32_t)(quad * 32) << 16) + acc * acc_stride;
      if constexpr (is_ozaki(MODE) && GEMM_EPI_GROUPS == 2) {
        if (NBUF == 1) {
          // One accumulator set: copy it to registers as (hi, lo) pairs and
          // release it before the stores, so that the next tile's MMAs run
          // while this tile's G is written.  With N tiles of at most EPI_NT_LO32
          // columns lo stays FP32 (at most three 16-column chunks per warp);
          // a wider tile (at most EPI_CHUNKS chunks, checked on the host)
          // holds lo rounded to BF16, two per register: |lo| <= ulp(hi) / 2, so
          // the pair keeps 2^-33 of the value, far below the 2^-28 of the
          // exact-slice operands.
          constexpr int CH = LO32 ? EPI_NT_LO32 / (16 * GEMM_EPI_GROUPS) : EPI_CHUNKS, LW = LO32 ? 16 : 8;
          constexpr int CUBE1 = g_cube_floats(LO32 ? G_PAIR : G_MIXED);
          float hv[CH][16];
          uint32_t lp[CH][LW];
#pragma unroll
          for (int k = 0; k < CH; ++k) {
            const int c0 = 16 * chunk0 + 32 * k;
            if (c0 < C.NT) {
#pragma unroll
              for (int half = 0; half < 2; ++half) {  // 8 columns at a time: fewer live registers
                const int cc = c0 + 8 * half;
                float a2[8], a3[8], ar[8];
                ptx::tmem_ld8x3(tbase + cc, tbase + C.NT + cc, tbase + 2 * C.NT + cc, a2, a3, ar);
#pragma unroll
                for (int j = 0; j < 8; j += 2) {
                  float l2[2];
#pragma unroll
                  for (int q = 0; q < 2; ++q) {
                    float s, e;
                    two_sum(a2[j + q], a3[j + q], s, e);
                    const float lo = __fadd_rn(e, ar[j + q]);
                    const float hi = __fadd_rn(s, lo);
                    hv[k][8 * half + j + q] = hi * gscale;
                    l2[q] = __fsub_rn(lo, __fsub_rn(hi, s)) * gscale;
                  }
                  if constexpr (LO32) {
                    lp[k][8 * half + j] = __float_as_uint(l2[0]);
                    lp[k][8 * half + j + 1] = __float_as_uint(l2[1]);
                  } else {
                    const __nv_bfloat162 b = __floats2bfloat162_rn(l2[0], l2[1]);
                    lp[k][4 * half + (j >> 1)] = *reinterpret_cast<const uint32_t*>(&b);
                  }
                }
              }
            }
          }
          ptx::tc_fence_before();
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive_cluster(ptx::mapa(&tempty[acc], 0));
          acc_phase ^= 1u;
          if (!valid) continue;
#pragma unroll
          for (int k = 0; k < CH; ++k) {
            const int c0 = 16 * chunk0 + 32 * k;
            if (c0 < C.NT) {
              const int z = c.z0 + c0;  // multiple of 16: two whole Z blocks
#pragma unroll
              for (int h2 = 0; h2 < 2; ++h2) {
                const int Z = (z >> 3) + h2;
                if (Z < nb) {
                  int64_t bt;
                  unsigned mask;
                  orbit_slots(x >> 3, y >> 3, Z, &bt, &mask);
                  xor_permute8(hv[k] + 8 * h2, zx);
                  float lv[LO32 ? 8 : 1];
                  uint4 l8 = make_uint4(0u, 0u, 0u, 0u);
                  if constexpr (LO32) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) lv[j] = __uint_as_float(lp[k][8 * h2 + j]);
                    xor_permute8(lv, zx);
                  } else {
                    l8 = xor_permute8_packed(lp[k] + 4 * h2, zx);
                  }
                  float* item = gslot + (bt * 18 + c.g * 6) * CUBE1;
                  for (int pid = 0; pid < 6; ++pid) {
                    if (!((mask >> pid) & 1u)) continue;
                    float* cube = item + pid * CUBE1;
                    store8(cube + roff, hv[k] + 8 * h2);
                    if constexpr (LO32) store8(cube + 512 + roff, lv);
                    else *reinterpret_cast<uint4*>(reinterpret_cast<unsigned short*>(cube + 512) + roff) = l8;
                  }
                }
              }
            }
          }
          continue;
        }
      }
      for (int c0 = 16 * chunk0; c0 < C.NT; c0 += 16 * GEMM_EPI_GROUPS) {
        const int z = c.z0 + c0;  // multiple of 16: two whole Z blocks
        if constexpr (is_ozaki(MODE)) {
          float a2[16], a3[16], ar[16];
          ptx::tmem_ld16x3(tbase + c0, tbase + C.NT + c0, tbase + 2 * C.NT + c0, a2, a3, ar);
          if (valid) {
            float hv[16], lv[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              float s, e;
              two_sum(a2[j], a3[j], s, e);
              const float lo = __fadd_rn(e, ar[j]);
              const float hi = __fadd_rn(s, lo);
              hv[j] = hi * gscale;
              lv[j] = __fsub_rn(lo, __fsub_rn(hi, s)) * gscale;
            }
#pragma unroll
            for (int h2 = 0; h2 < 2; ++h2) {
              const int Z = (z >> 3) + h2;
              if (Z < nb) {
                int64_t bt;
                unsigned mask;
                orbit_slots(x >> 3, y >> 3, Z, &bt, &mask);
                xor_permute8(hv + 8 * h2, zx);
                xor_permute8(lv + 8 * h2, zx);
                float* item = gslot + (bt * 18 + c.g * 6) * CUBE;
                for (int pid = 0; pid < 6; ++pid) {
                  if (!((mask >> pid) & 1u)) continue;
                  float* cube = item + pid * CUBE;
                  store8(cube + roff, hv + 8 * h2);
                  store8(cube + 512 + roff, lv + 8 * h2);
                }
              }
            }
          }
        } else {
          float vals[16];
          ptx::tmem_ld16(tbase + c0, vals);
          if (valid) {
#pragma unroll
            for (int h2 = 0; h2 < 2; ++h2) {
              const int Z = (z >> 3) + h2;
              if (Z < nb) {
                int64_t bt;
                unsigned mask;
                orbit_slots(x >> 3, y >> 3, Z, &bt, &mask);
                xor_permute8(vals + 8 * h2, zx);
                float* item = gslot + (bt * 18 + c.g * 6) * 512;
                for (int pid = 0; pid < 6; ++pid)
                  if ((mask >> pid) & 1u) store8(item + pid * 512 + roff, vals + 8 * h2);
              }
            }
          }
        }
      }
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive_cluster(ptx::mapa(&tempty[acc], 0));
      if (NBUF == 2) {
        acc ^= 1u;
        if (acc == 0) acc_phase ^= 1u;
      } else {
        acc_phase ^= 1u;
      }
    }
  }

  __syncwarp();
  ptx::tc_fence_before();
  __syncthreads();
  ptx::cluster_sync();  // neither CTA leaves while the other's MMAs or signals may reach it
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc_pair(tmem_base, P.tmem_cols);
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

struct TcState {
  PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
};

static TcState* tc_state(Handle* h) {
  if (!h->tc) h->tc = new TcState();
  return static_cast<TcState*>(h->tc);
}

void destroy_tc_state(Handle* h) {
  delete static_cast<TcState*>(h->tc);
  h->tc = nullptr;
}

static te_status get_encoder(TcState* st) {
  if (st->encode) return TE_OK;
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
          cudaSuccess ||
      q != cudaDriverEntryPointSuccess || !fn) {
    cudaGetLastError();
    return fail(TE_ECUDA, "cuTensorMapEncodeTiled entry point not available");
  }
  st->encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  return TE_OK;
}

struct TcPlan {
  int mode, es, nparts, fmt;  // fmt: G format
  int vp, op, vq;
  int TA, TB, NT, n_my, n_mp, n_nt;
  int kw_chunks, ko_chunks, kw_elems, ko_elems, cbw, cbo;
  int stages;
  uint32_t stage_bytes, tmem_cols;
  int nbuf;
  int nslots, par_slots;  // triples per launch, and per share reduction
  int min_slots;          // triples per launch where memory is short
};

constexpr int64_t MIN_SLOTS = 4;          // triples per launch where memory is short,
constexpr int64_t MIN_POOL = int64_t(3) << 30;  // as many as this holds
// Triples whose energy partials wait for one share reduction (about 20 MB of
// them) where memory is not short; a launch's own triples where it is.
constexpr int64_t TC_PAR_SLOTS = 1024;

static int round_up(int x, int m) { return (x + m - 1) / m * m; }

static TcPlan make_plan(const Handle* h, int o, int v, int mode, int64_t ntri, int force_tb = 0,
                        int force_nnt = 0) {
  TcPlan pl{};
  pl.mode = mode;
  const bool oz = is_ozaki(mode);
  pl.es = (mode == TC_BF16X3 || oz) ? 2 : 4;
  pl.nparts = mode == TC_TF32 ? 1 : (mode == TC_OZAKI ? 4 : (mode == TC_OZAKI6 ? 5 : 2));
  const int nacc = oz ? 3 : 1;
  // TF32/BF16X3 (one accumulator) double-buffer at any N tile; the exact-slice
  // modes (three accumulators) take N tiles up to 160 single-buffered, and
  // double-buffer when 2 x 3 x NT <= 512 columns (NT <= 64, in steps of 32)
  const int nbuf_max = oz ? 1 : 2;
  pl.vp = round_up(v, 16);
  pl.op = round_up(o, 16);
  pl.vq = round_up(v, 4);
  // M tile: TA x-values by TB y-values, TA*TB = 128, least padding
  int bestTB = 128;
  int64_t best = -1;
  for (int TB = 128; TB >= 16; TB /= 2) {
    const int TA = 128 / TB;
    const int64_t rows = (int64_t)round_up(v, TA) * round_up(v, TB);
    if (best < 0 || rows < best) {
      best = rows;
      bestTB = TB;
    }
  }
  const int defTB = bestTB;
  if (!force_tb) {
    auto it = h->tuned.find(std::make_tuple(o, v, mode));
    if (it != h->tuned.end()) {
      force_tb = it->second.first;
      force_nnt = it->second.second;
    }
  }
  if (force_tb) bestTB = force_tb;
  pl.TB = bestTB;
  pl.TA = 128 / bestTB;
  pl.n_my = (v + pl.TB - 1) / pl.TB;
  pl.n_mp = ((v + pl.TA - 1) / pl.TA * pl.n_my + 1) / 2;
  const int ntmax = std::min(256, (512 / (nacc * nbuf_max)) / 32 * 32);
  const int def_nt = pl.n_nt = (v + ntmax - 1) / ntmax;
  // a tuned split: any count whose N tile fits three accumulators in TMEM (N <= 160)
  if (force_nnt > 0 && round_up((v + force_nnt - 1) / force_nnt, 32) <= (oz ? 160 : 256)) pl.n_nt = force_nnt;
  pl.NT = round_up((v + pl.n_nt - 1) / pl.n_nt, 32);  // cta_group::2: N in steps of 32
  pl.nbuf = (2 * nacc * pl.NT <= 512) ? 2 : 1;
  // G's low words stay FP32 in tiles of at most 80 columns (two accumulator sets
  // up to 64, one set and three chunks per epilogue warp above), also where the
  // step of 32 pads the tile to 96; wider tiles round them to BF16.
  auto format = [&](int n_nt) { return !oz ? G_F32 : ((v + n_nt - 1) / n_nt <= 80 ? G_PAIR : G_MIXED); };
  pl.fmt = format(pl.n_nt);
  pl.cbw = oz ? 64 : 128;
  pl.kw_elems = pl.cbw / pl.es;
  pl.kw_chunks = (pl.vp + pl.kw_elems - 1) / pl.kw_elems;
  const int obytes = pl.op * pl.es;
  pl.cbo = obytes <= 32 ? 32 : (obytes <= 64 ? 64 : std::min(128, pl.cbw));
  pl.ko_elems = pl.cbo / pl.es;
  pl.ko_chunks = (pl.op + pl.ko_elems - 1) / pl.ko_elems;
  // 128 rows of A and this CTA's half of the B tile, every part
  pl.stage_bytes = (uint32_t)pl.nparts * (128u + (uint32_t)(pl.NT / 2)) * (uint32_t)pl.cbw;
  const size_t avail = h->smem_optin > 2048 ? h->smem_optin - 2048 : 0;
  pl.stages = (int)std::min<size_t>(8, avail / pl.stage_bytes);
  uint32_t cols = 32;
  while (cols < (uint32_t)(nacc * pl.nbuf * pl.NT)) cols <<= 1;
  pl.tmem_cols = cols;
  // pair tiles and G bytes per triple in the default shape; a tuned one gets the G
  // pool that this makes, so that the workspace does not depend on the tuning
  const int64_t def_m = (int64_t)((v + 128 / defTB - 1) / (128 / defTB)) * ((v + defTB - 1) / defTB);
  const int64_t tiles = 3LL * ((def_m + 1) / 2) * def_nt;
  const int64_t def_slot = g_slot_floats(v, format(def_nt)) * 4, per_slot = g_slot_floats(v, pl.fmt) * 4;
  // About 40 tiles per pair of CTAs and launch: a launch's fixed part (its
  // first loads, the last tile's epilogue, a last wave) is some 15 us, which at
  // nvir = 120 with four triples per launch was a sixth of the contraction
  // (nocc=16 nvir=120 energy: 33.9 ms with 4 triples per launch, 30.5 with 9,
  // 29.1 with 17).
  int64_t want = (20LL * std::max(1, h->num_sms) + tiles - 1) / tiles;
  const int64_t mem_cap = std::max<int64_t>(1, (int64_t)(6LL << 30) / def_slot);
  want = std::max<int64_t>(want, MIN_SLOTS);
  want = std::max<int64_t>(1, std::min<int64_t>({want, mem_cap, 1024, ntri}));
  auto fit = [&](int64_t slots) { return (int)std::max<int64_t>(1, std::min<int64_t>(slots, slots * def_slot / per_slot)); };
  pl.nslots = fit(want);
  pl.par_slots = (int)std::max<int64_t>(pl.nslots, std::min<int64_t>(TC_PAR_SLOTS, ntri));
  // at the least, a tile for every pair of CTAs
  const int64_t fill = (std::max(1, h->num_sms) / 2 + tiles - 1) / tiles;
  pl.min_slots = fit(std::max<int64_t>(1, std::min<int64_t>({want, std::max(MIN_SLOTS, fill), MIN_POOL / def_slot})));
  return pl;
}

// ---------------------------------------------------------------------------
// host side: workspace, launch rounds
// ---------------------------------------------------------------------------

// One cluster's part of the workspace: the operand planes, the float32
// copies the energy kernel reads, the scale exponents and the per-triple
// shares.  The G pool and the energy partials are shared by a whole run.
struct TcBuffers {
  void *a[MAX_PARTS], *b[MAX_PARTS], *l[MAX_PARTS], *n[MAX_PARTS];
  float *ovs32, *t1_32;
  double* etri;
  unsigned int* maxhi;  // high words of max |ovvv|, |t2|, |ooov|
  int* exps;
};

static size_t tc_carve_cluster(char* base, const TcPlan& pl, int64_t o, int64_t v, int64_t ntri, TcBuffers* b) {
  size_t off = 0;
  auto take = [&](size_t bytes) -> void* {
    off = (off + 1023) & ~size_t(1023);
    void* p = base ? base + off : nullptr;
    off += bytes;
    return p;
  };
  const size_t es = (size_t)pl.es;
  const size_t na = (size_t)o * v * v * pl.vp, nb = (size_t)o * o * v * pl.vp;
  const size_t nl = (size_t)o * v * v * pl.op, nn = (size_t)o * o * v * pl.op;
  // one slice-interleaved block per array; part k points at slice k of the
  // first row group (groups: v^2 rows per occupied index for ovvv and t2L,
  // v rows per occupied pair for t2 and nooT)
  const size_t ns = (size_t)pl.nparts;
  char* A = static_cast<char*>(take(ns * na * es));
  char* B = static_cast<char*>(take(ns * nb * es));
  char* Lb = static_cast<char*>(take(ns * nl * es));
  char* Nb = static_cast<char*>(take(ns * nn * es));
  for (int k = 0; k < MAX_PARTS; ++k) {
    const bool use = k < pl.nparts && base;
    b->a[k] = use ? A + (size_t)k * v * v * pl.vp * es : nullptr;
    b->b[k] = use ? B + (size_t)k * v * pl.vp * es : nullptr;
    b->l[k] = use ? Lb + (size_t)k * v * v * pl.op * es : nullptr;
    b->n[k] = use ? Nb + (size_t)k * v * pl.op * es : nullptr;
  }
  b->ovs32 = static_cast<float*>(take((size_t)o * v * o * pl.vq * 4));
  b->t1_32 = static_cast<float*>(take((size_t)o * pl.vq * 4));
  b->etri = static_cast<double*>(take((size_t)std::max<int64_t>(1, ntri) * 8));
  b->maxhi = static_cast<unsigned int*>(take(4 * 4));
  b->exps = static_cast<int*>(take(8 * 4));
  return (off + 1023) & ~size_t(1023);
}

// Workspace of one run: the clusters' parts, then the G pool, then the
// energy partials: per triple, one float64 sum per block (one block per SM)
// and compute warp, for the rounds up to the next share reduction.
struct TcPool {
  int64_t pool_floats;
  int64_t max_slots;  // G slots per launch
  int64_t par_slots;  // energy partials held until their share reduction (at least max_slots)
};

static size_t tc_partial_bytes(const TcPool& q, int num_sms) {
  return (size_t)q.par_slots * std::max(1, num_sms) * ENERGY_TC_WARPS * sizeof(double);
}

static size_t tc_shared_bytes(const TcPool& q, int num_sms) {
  const size_t g = ((size_t)q.pool_floats * 4 + 1023) & ~size_t(1023);
  return g + tc_partial_bytes(q, num_sms) + 1024;
}

static te_status encode(TcState* st, CUtensorMap* m, const void* base, CUtensorMapDataType dt, int rank,
                        const uint64_t* dims, const uint64_t* strides_bytes, const uint32_t* box,
                        CUtensorMapSwizzle swz, const char* what) {
  cuuint64_t gd[5];
  cuuint64_t gs[4];
  cuuint32_t bd[5], e1[5];
  for (int i = 0; i < rank; ++i) {
    gd[i] = dims[i];
    bd[i] = box[i];
    e1[i] = 1;
    if (i < rank - 1) gs[i] = strides_bytes[i];
  }
  CUresult r = st->encode(m, dt, (cuuint32_t)rank, const_cast<void*>(base), gd, gs, bd, e1,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(TE_ECUDA, "tensor map encoding failed for %s (CUresult %d)", what, (int)r);
  return TE_OK;
}

static CUtensorMapSwizzle swz_of(int cb) {
  return cb == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : (cb == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
}

static te_status build_maps(TcState* st, const TcPlan& pl, int o, int v, const TcBuffers& b, TcMaps* M) {
  std::memset(M, 0, sizeof(*M));
  const CUtensorMapDataType dt = pl.es == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
  const uint64_t es = (uint64_t)pl.es;
  const uint64_t vp = pl.vp, op = pl.op, V = v, O = o, NS = (uint64_t)pl.nparts;
  const uint32_t ns = (uint32_t)pl.nparts;
  te_status s;
  {  // ovvv slices [p][s][x][y][d]: dims (d, y, x, s, p)
    const uint64_t d[5] = {vp, V, V, NS, O};
    const uint64_t sn[4] = {vp * es, V * vp * es, V * V * vp * es, NS * V * V * vp * es};
    const uint32_t box[5] = {(uint32_t)pl.kw_elems, (uint32_t)pl.TB, (uint32_t)pl.TA, ns, 1};
    if ((s = encode(st, &M->a_nat, b.a[0], dt, 5, d, sn, box, swz_of(pl.cbw), "ovvv")) != TE_OK) return s;
    // transposed rows: element (d, y, x, s, q) at ovvv[q][s][y][x][d]
    const uint64_t stt[4] = {V * vp * es, vp * es, V * V * vp * es, NS * V * V * vp * es};
    if ((s = encode(st, &M->a_tr, b.a[0], dt, 5, d, stt, box, swz_of(pl.cbw), "ovvv^T")) != TE_OK) return s;
  }
  {  // t2L slices [q][s][x][y][l]: dims (l, y, x, s, q)
    const uint64_t d[5] = {op, V, V, NS, O};
    const uint64_t sn[4] = {op * es, V * op * es, V * V * op * es, NS * V * V * op * es};
    const uint32_t box[5] = {(uint32_t)pl.ko_elems, (uint32_t)pl.TB, (uint32_t)pl.TA, ns, 1};
    if ((s = encode(st, &M->l_nat, b.l[0], dt, 5, d, sn, box, swz_of(pl.cbo), "t2L")) != TE_OK) return s;
    const uint64_t stt[4] = {V * op * es, op * es, V * V * op * es, NS * V * V * op * es};
    if ((s = encode(st, &M->l_tr, b.l[0], dt, 5, d, stt, box, swz_of(pl.cbo), "t2L^T")) != TE_OK) return s;
  }
  {  // t2 slices [r][q][s][z][d]: dims (d, z, s, q, r)
    const uint64_t d[5] = {vp, V, NS, O, O};
    const uint64_t sn[4] = {vp * es, V * vp * es, NS * V * vp * es, O * NS * V * vp * es};
    const uint32_t box[5] = {(uint32_t)pl.kw_elems, (uint32_t)pl.NT / 2, ns, 1, 1};
    if ((s = encode(st, &M->b_t2, b.b[0], dt, 5, d, sn, box, swz_of(pl.cbw), "t2")) != TE_OK) return s;
  }
  {  // nooT slices [p][r][s][z][l]: dims (l, z, s, r, p)
    const uint64_t d[5] = {op, V, NS, O, O};
    const uint64_t sn[4] = {op * es, V * op * es, NS * V * op * es, O * NS * V * op * es};
    const uint32_t box[5] = {(uint32_t)pl.ko_elems, (uint32_t)pl.NT / 2, ns, 1, 1};
    if ((s = encode(st, &M->b_noo, b.n[0], dt, 5, d, sn, box, swz_of(pl.cbo), "nooT")) != TE_OK) return s;
  }
  return TE_OK;
}

struct EnergyMapsHost {
  CUtensorMap ovs, t1;
};

static te_status build_energy_maps(TcState* st, const TcPlan& pl, int o, int v, const TcBuffers& b,
                                   EnergyMapsHost* E) {
  std::memset(E, 0, sizeof(*E));
  const uint64_t V = v, O = o, vq = pl.vq;
  te_status s;
  {  // ovs32 [i][a][j][vq]: dims (b, j, a, i)
    const uint64_t d[4] = {V, O, V, O};
    const uint64_t sn[3] = {vq * 4, O * vq * 4, V * O * vq * 4};
    const uint32_t box[4] = {8, 1, 8, 1};
    if ((s = encode(st, &E->ovs, b.ovs32, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, d, sn, box,
                    CU_TENSOR_MAP_SWIZZLE_NONE, "ovs")) != TE_OK)
      return s;
  }
  {  // t1 [i][vq]: dims (a, i)
    const uint64_t d[2] = {V, O};
    const uint64_t sn[1] = {vq * 4};
    const uint32_t box[2] = {8, 1};
    if ((s = encode(st, &E->t1, b.t1_32, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, d, sn, box,
                    CU_TENSOR_MAP_SWIZZLE_NONE, "t1")) != TE_OK)
      return s;
  }
  return TE_OK;
}

// ---------------------------------------------------------------------------
// ovvv from density-fitting factors (t_energy_df):
//   ovvv[p,x,y,d] = sum_P Bov[P,p,x] Bvv[P,y,d]
// formed nst slabs at a time by the exact-slice view GEMM (five 7-bit slices
// per factor, K in exact blocks of 128) into a float64 staging block,
// then cut into the contraction's operand form.
// ---------------------------------------------------------------------------

constexpr int DF_NS = 5;                                  // slices per factor
constexpr size_t DF_STAGE_BYTES = size_t(2) << 30;        // staging block limit

// Scratch of the formation.  It shares the region of the G pool, which the
// contraction only writes after every operand is ready (stream order).
struct DfScratch {
  __nv_bfloat16 *bov = nullptr, *bvv = nullptr;  // DF_NS planes each, [p, x][Pp] and [y, d][Pp]
  unsigned int* mx = nullptr;                    // max |Bov|, max |Bvv| (high words)
  int* ex = nullptr;                             // their scale exponents
  double* stage = nullptr;                       // nst slabs of v^3
  int nst = 0;
};

static int64_t df_pitch(int64_t naux) { return (naux + 7) / 8 * 8; }  // tensor-map rows in steps of 16 bytes

static size_t df_carve(char* base, int o, int v, int64_t naux, DfScratch* d) {
  size_t off = 0;
  auto take = [&](size_t bytes) -> char* {
    off = (off + 1023) & ~size_t(1023);
    char* p = base ? base + off : nullptr;
    off += bytes;
    return p;
  };
  const size_t v3 = (size_t)v * v * v;
  d->nst = (int)std::max<size_t>(1, std::min<size_t>((size_t)o, DF_STAGE_BYTES / (v3 * 8)));
  d->bov = reinterpret_cast<__nv_bfloat16*>(take((size_t)DF_NS * df_pitch(naux) * o * v * 2));
  d->bvv = reinterpret_cast<__nv_bfloat16*>(take((size_t)DF_NS * df_pitch(naux) * v * v * 2));
  d->mx = reinterpret_cast<unsigned int*>(take(16));
  d->ex = reinterpret_cast<int*>(take(8));
  d->stage = reinterpret_cast<double*>(take((size_t)d->nst * v3 * 8));
  return (off + 1023) & ~size_t(1023);
}

// slabs p0 .. p0+ne-1 of ovvv into the staging block ([p - p0][x][y][d])
static te_status df_form(Handle* h, const te_df* df, int o, int v, int p0, int ne, const DfScratch& d, cudaStream_t s) {
  const int64_t Pp = df_pitch(df->naux), ov = (int64_t)o * v, vv = (int64_t)v * v;
  return vt_product(h, d.bov + (int64_t)p0 * v * Pp, ov * Pp, (int64_t)ne * v, d.bvv, vv * Pp, vv, df->naux, Pp, DF_NS, d.ex,
                    d.ex + 1, d.stage, s);
}

// Operand planes of one cluster: one pass over the inputs for the value
// checks (err set) and the largest magnitudes, then one launch that cuts every
// operand.  With df, ovvv comes from the factors (the slabs are formed once
// for the maximum in the exact-slice modes, once for the slices: the same bits
// both times); else from c->ovvv.
static te_status launch_prep_tc(Handle* h, int mode, const te_cluster* c, const TcPlan& pl, const TcBuffers& b,
                                  const te_df* df, const DfScratch* dfs, unsigned int* err, int64_t cluster,
                                  cudaStream_t s) {
  auto bad = [](cudaError_t e) { return fail(TE_ECUDA, "operand split launch: %s", cudaGetErrorString(e)); };
  const int num_sms = h->num_sms;
  int64_t* const launches = &h->n_launches;
  const int o = (int)c->nocc, v = (int)c->nvir;
  const int64_t v2 = (int64_t)v * v, v3 = v2 * v;
  const bool oz = is_ozaki(mode);
  cudaError_t e = cudaSuccess;
  if (oz || df || err) {
    MaxOut mo{};
    if (oz) {
      mo.ovvv = df ? nullptr : b.maxhi;
      mo.t2 = b.maxhi + 1;
      mo.ooov = b.maxhi + 2;
      if ((e = cudaMemsetAsync(b.maxhi, 0, 4 * 4, s)) != cudaSuccess) return bad(e);
    }
    if (df) {
      mo.bov = dfs->mx;
      mo.bvv = dfs->mx + 1;
      if ((e = cudaMemsetAsync(dfs->mx, 0, 2 * 4, s)) != cudaSuccess) return bad(e);
    }
    e = launch_check_inputs(c, cluster, err, num_sms, s, df, &mo);
    ++*launches;
    if (e != cudaSuccess) return bad(e);
  }
  if (df) {
    const int64_t P = df->naux, Pp = df_pitch(P);
    e = slice_rows(df->Bov, (int64_t)o * v, P, Pp, DF_NS, dfs->mx, dfs->ex, dfs->bov, s, launches);
    if (e == cudaSuccess) e = slice_rows(df->Bvv, v2, P, Pp, DF_NS, dfs->mx + 1, dfs->ex + 1, dfs->bvv, s, launches);
    for (int p0 = 0; oz && p0 < o && e == cudaSuccess; p0 += dfs->nst) {
      const int ne = std::min(dfs->nst, o - p0);
      const te_status st = df_form(h, df, o, v, p0, ne, *dfs, s);
      if (st != TE_OK) return st;
      const MaxArray a{dfs->stage, 1, (int64_t)ne * v3, 0, b.maxhi, nullptr, 0, 0u};
      e = launch_absmax(&a, 1, nullptr, 0, nullptr, 0, 0, nullptr, num_sms, s);
      ++*launches;
    }
    if (e != cudaSuccess) return bad(e);
  }
  SplitScales sc{};
  if (oz) {
    sc.maxhi = b.maxhi;
    sc.exps = b.exps;
  }
  auto parts = [](void* const* p) { return Parts{{p[0], p[1], p[2], p[3], p[4]}}; };
  const int64_t ov = (int64_t)o * v;
  SplitJob jobs[SPLIT_MAX_JOBS] = {};
  int n = 0;
  if (!df) jobs[n++] = SplitJob{SPLIT_ROWS, c->ovvv, parts(b.a), nullptr, v, pl.vp, o * v2, 1, 0, 0, v2, 1, 0, nullptr, 0};
  jobs[n++] = SplitJob{SPLIT_ROWS, c->t2, parts(b.b), nullptr, v, pl.vp, (int64_t)o * o * v, 1, 0, 0, v, 1, 1, nullptr, 0};
  // t2L[q][x][y][l] = t2[l,q,x,y]; nooT[p][r][z][l] = -ooov[p,l,r,z]
  jobs[n++] = SplitJob{SPLIT_COLS, c->t2, parts(b.l), nullptr, o, pl.op, v2, o, v2, o * v2, v2, 1, 2, nullptr, 0};
  jobs[n++] = SplitJob{SPLIT_COLS, c->ooov, parts(b.n), nullptr, o, pl.op, ov, o, o * ov, ov, v, -1, 3, nullptr, 0};
  jobs[n++] = SplitJob{SPLIT_OVS, c->ovov, Parts{}, b.ovs32, v, pl.vq, o, 1, 0, 0, 1, 1, 0, nullptr, 0};
  jobs[n++] = SplitJob{SPLIT_COPY, c->t1, Parts{}, b.t1_32, v, pl.vq, o, 1, 0, 0, 1, 1, 0, nullptr, 0};
  e = launch_split(mode, jobs, n, sc, s);
  ++*launches;
  // one occupied index's slices of ovvv: nparts consecutive [v^2][vp] blocks
  const size_t group = (size_t)pl.nparts * v2 * pl.vp * pl.es;
  for (int p0 = 0; df && p0 < o && e == cudaSuccess; p0 += dfs->nst) {
    const int ne = std::min(dfs->nst, o - p0);
    const te_status st = df_form(h, df, o, v, p0, ne, *dfs, s);
    if (st != TE_OK) return st;
    Parts Ap{};
    for (int k = 0; k < MAX_PARTS; ++k) Ap.p[k] = b.a[k] ? static_cast<char*>(b.a[k]) + (size_t)p0 * group : nullptr;
    const SplitJob slab{SPLIT_ROWS, dfs->stage, Ap, nullptr, v, pl.vp, ne * v2, 1, 0, 0, v2, 1, 0, nullptr, 0};
    e = launch_split(mode, &slab, 1, sc, s);
    ++*launches;
  }
  return e == cudaSuccess ? TE_OK : bad(e);
}

template <int MODE, bool LO32 = false>
static cudaError_t launch_gemm_tc(const TcMapSet& M, const TcParams& P, size_t smem, int grid_cap, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(k_gemm_tc<MODE, LO32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int64_t grid = GEMM_PAIR * std::min<int64_t>(P.total_tiles, std::max(1, grid_cap / GEMM_PAIR));
  k_gemm_tc<MODE, LO32><<<(unsigned)grid, GEMM_THREADS, smem, s>>>(M, P);
  return cudaGetLastError();
}

static cudaError_t launch_gemm_any(int mode, const TcMapSet& M, const TcParams& P, size_t smem, int grid_cap,
                                   cudaStream_t s) {
  if (mode == TC_BF16X3) return launch_gemm_tc<TC_BF16X3>(M, P, smem, grid_cap, s);
  if (mode == TC_TF32X3) return launch_gemm_tc<TC_TF32X3>(M, P, smem, grid_cap, s);
  if (mode == TC_TF32) return launch_gemm_tc<TC_TF32>(M, P, smem, grid_cap, s);
  const bool lo32 = P.fmt == G_PAIR;
  if (mode == TC_OZAKI)
    return lo32 ? launch_gemm_tc<TC_OZAKI, true>(M, P, smem, grid_cap, s) : launch_gemm_tc<TC_OZAKI>(M, P, smem, grid_cap, s);
  return lo32 ? launch_gemm_tc<TC_OZAKI6, true>(M, P, smem, grid_cap, s) : launch_gemm_tc<TC_OZAKI6>(M, P, smem, grid_cap, s);
}

// One cluster of a run: its plan, buffers, tensor maps and triple range.
struct TcJob {
  const te_cluster* c = nullptr;
  TcPlan pl{};
  TcBuffers b{};
  TcMaps maps{};
  EnergyMapsHost em{};
  int o = 0, v = 0;
  int64_t t_begin = 0, t_end = 0;
  int64_t nbt = 0, slot_floats = 0, tiles_per_triple = 0;
  double* shares = nullptr;  // share of triple t at shares[t - t_begin]
  double* e_out = nullptr;   // sum of the shares (nullable)
};

static void fill_cluster(const TcJob& J, TcCl* C) {
  C->o = J.o;
  C->v = J.v;
  C->TA = J.pl.TA;
  C->TB = J.pl.TB;
  C->NT = J.pl.NT;
  C->n_my = J.pl.n_my;
  C->n_mp = J.pl.n_mp;
  C->n_nt = J.pl.n_nt;
  C->kw_chunks = J.pl.kw_chunks;
  C->ko_chunks = J.pl.ko_chunks;
  C->kw_elems = J.pl.kw_elems;
  C->ko_elems = J.pl.ko_elems;
  C->cbo = J.pl.cbo;
  C->slot_floats = J.slot_floats;
  C->exps = J.b.exps;
}

// Contraction parameters of one launch over the clusters jl[0..ncl) of `jobs`
// and the given pieces; *smem receives the dynamic shared memory.
static te_status gemm_params(const Handle* h, const std::vector<TcJob>& jobs, const int* jl, int ncl,
                             const TcPiece* pcs, int npieces, int64_t tiles, int mode, TcParams* P, TcMapSet* M,
                             size_t* smem) {
  std::memset(P, 0, sizeof(*P));
  std::memset(M, 0, sizeof(*M));
  uint32_t stage_max = 0;
  int nt_max = 0;
  for (int q = 0; q < ncl; ++q) {
    const TcJob& J = jobs[jl[q]];
    fill_cluster(J, &P->cl[q]);
    M->m[q] = J.maps;
    stage_max = std::max(stage_max, J.pl.stage_bytes);
    nt_max = std::max(nt_max, J.pl.NT);
  }
  const TcPlan& p0 = jobs[jl[0]].pl;
  const int nacc = is_ozaki(mode) ? 3 : 1;
  P->ncl = ncl;
  P->npieces = npieces;
  P->cbw = p0.cbw;
  P->a_part_bytes = 128u * (uint32_t)p0.cbw;
  P->stage_bytes = stage_max;
  const size_t avail = h->smem_optin > 2048 ? h->smem_optin - 2048 : 0;
  P->stages = (int)std::min<size_t>(8, avail / stage_max);
  if (P->stages < 2) return fail(TE_EUNSUPPORTED, "not enough shared memory for two pipeline stages");
  P->nbuf = p0.nbuf;
  P->fmt = p0.fmt;
  P->nt_max = nt_max;
  const int nt_held = P->fmt == G_PAIR ? EPI_NT_LO32 : EPI_NT_MAX;
  if (is_ozaki(mode) && P->nbuf == 1 && nt_max > nt_held)
    return fail(TE_EUNSUPPORTED, "N tile %d above the epilogue's %d columns", nt_max, nt_held);
  uint32_t cols = 32;
  while (cols < (uint32_t)(nacc * P->nbuf * nt_max)) cols <<= 1;
  P->tmem_cols = cols;
  P->total_tiles = tiles;
  P->triples = h->d_triples;
  P->err = h->d_err;
  P->wait_ns = h->wait_limit_ns;
  for (int q = 0; q < npieces; ++q) P->pc[q] = pcs[q];
  *smem = (size_t)P->stages * stage_max + 1024 + 256;
  return TE_OK;
}

// Runs the jobs' triples in rounds: each round fills the G pool with pieces
// (up to TC_MAX_CL clusters, TC_MAX_PIECES pieces, one TMEM buffering and G format), then
// launches the contraction and the energy epilogue once.  The shares are
// reduced when the partials of par_slots triples or TC_MAX_PIECES runs of
// triples have come together, and at the end; then each job's total.  Pieces
// follow the jobs' order.
static te_status run_rounds(Handle* h, std::vector<TcJob>& jobs, int mode, float* pool, const TcPool& pq,
                            double* partials, cudaStream_t s) {
  const double nprod = (mode == TC_TF32) ? 1.0 : (mode == TC_OZAKI ? 10.0 : (mode == TC_OZAKI6 ? 15.0 : 3.0));
  size_t j = 0;
  int64_t t = jobs.empty() ? 0 : jobs[0].t_begin;
  std::vector<TcPiece> pcs;
  TcMapSet* MS = new TcMapSet;
  TcParams* P = new TcParams;
  EnergyLaunch* EL = new EnergyLaunch;
  te_status st = TE_OK;
  const int egrid = (int)energy_tc_grid(h->num_sms);
  std::vector<TcPiece> held;  // runs of triples whose partials wait for the share reduction
  int nheld = 0;              // their slots
  auto reduce_held = [&]() {
    if (held.empty()) return;
    const cudaError_t e = launch_reduce_pieces(partials, egrid, h->d_triples, held.data(), (int)held.size(), nheld, s);
    ++h->n_launches;
    if (e != cudaSuccess) st = fail(TE_ECUDA, "share reduction launch: %s", cudaGetErrorString(e));
    held.clear();
    nheld = 0;
  };
  while (st == TE_OK) {
    while (j < jobs.size() && t >= jobs[j].t_end) {
      ++j;
      if (j < jobs.size()) t = jobs[j].t_begin;
    }
    if (j >= jobs.size()) break;
    int jl[TC_MAX_CL];
    int ncl = 0, nbuf = -1, fmt = 0, nslots = 0;
    int64_t used = 0, tiles = 0;
    double flops = 0.0;
    pcs.clear();
    while (j < jobs.size() && (int)pcs.size() < TC_MAX_PIECES) {
      TcJob& J = jobs[j];
      if (t >= J.t_end) {
        ++j;
        if (j < jobs.size()) t = jobs[j].t_begin;
        continue;
      }
      int cl = -1;
      for (int q = 0; q < ncl; ++q)
        if (jl[q] == (int)j) cl = q;
      if (cl < 0) {
        if (ncl == TC_MAX_CL || (nbuf >= 0 && (J.pl.nbuf != nbuf || J.pl.fmt != fmt))) break;
        cl = ncl;
      }
      const int64_t fit = std::min((pq.pool_floats - used) / J.slot_floats, pq.max_slots - nslots);
      if (fit <= 0) break;
      if (cl == ncl) {
        jl[ncl++] = (int)j;
        nbuf = J.pl.nbuf;  // one TMEM buffering and one G format per launch
        fmt = J.pl.fmt;
      }
      const int ns = (int)std::min<int64_t>(fit, J.t_end - t);
      TcPiece pc{};
      pc.cl = cl;
      pc.ns = ns;
      pc.slot0 = nslots;
      pc.t0 = t;
      pc.tile0 = tiles;
      pc.nbt = J.nbt;
      pc.gbuf = pool + used;
      pc.shares = J.shares + (t - J.t_begin);
      pcs.push_back(pc);
      used += (int64_t)ns * J.slot_floats;
      nslots += ns;
      tiles += (int64_t)ns * J.tiles_per_triple;
      t += ns;
      const double kpad = 2.0 * J.pl.kw_chunks * J.pl.kw_elems + 2.0 * J.pl.ko_chunks * J.pl.ko_elems;
      flops += 2.0 * nprod * (double)ns * J.tiles_per_triple * 256.0 * J.pl.NT * kpad;
    }
    if (pcs.empty()) {
      st = fail(TE_ENOMEM, "G pool smaller than one triple's G blocks");
      break;
    }
    if (nheld + nslots > pq.par_slots || held.size() + pcs.size() > (size_t)TC_MAX_PIECES) reduce_held();
    if (st != TE_OK) break;
    for (const TcPiece& pc : pcs) {
      // a run that continues the last one (same cluster, next triple) joins it
      if (!held.empty() && held.back().shares + held.back().ns == pc.shares && held.back().t0 + held.back().ns == pc.t0 &&
          held.back().nbt == pc.nbt) {
        held.back().ns += pc.ns;
      } else {
        held.push_back(pc);
        held.back().slot0 = nheld + pc.slot0;
      }
    }
    size_t smem = 0;
    st = gemm_params(h, jobs, jl, ncl, pcs.data(), (int)pcs.size(), tiles, mode, P, MS, &smem);
    if (st != TE_OK) break;
    std::memset(EL, 0, sizeof(*EL));
    EL->ncl = ncl;
    EL->npieces = (int)pcs.size();
    EL->fmt = jobs[jl[0]].pl.fmt;
    EL->num_sms = h->num_sms;
    for (int q = 0; q < ncl; ++q) {
      const TcJob& J = jobs[jl[q]];
      EL->cl[q] = EnergyCl{J.o, J.v, (int)energy_num_blocks(J.v), J.nbt, J.c->eps_o, J.c->eps_v};
      EL->map_ovs[q] = &J.em.ovs;
      EL->map_t1[q] = &J.em.t1;
    }
    for (size_t q = 0; q < pcs.size(); ++q) EL->pc[q] = pcs[q];
    EL->triples = h->d_triples;
    EL->partials = partials + (int64_t)nheld * egrid * ENERGY_TC_WARPS;
    nheld += nslots;
    EL->err = h->d_err;
    EL->wait_ns = h->wait_limit_ns;
    if (h->log)
      std::fprintf(stderr, "[tenergy] round: %d clusters, %zu pieces, %d triples, %lld tiles\n",
                   ncl, pcs.size(), nslots, (long long)tiles);
    size_t pm = prof_begin(h, 0, s);
    cudaError_t e = launch_gemm_any(mode, *MS, *P, smem, h->num_sms, s);
    prof_end(h, pm, s);
    h->gemm_flops += flops;
    if (e == cudaSuccess) {
      pm = prof_begin(h, 1, s);
      e = launch_energy_tc(*EL, s);
      prof_end(h, pm, s);
    }
    h->n_launches += 2;
    if (e != cudaSuccess) st = fail(TE_ECUDA, "tensor-core path launch: %s", cudaGetErrorString(e));
  }
  if (st == TE_OK) reduce_held();
  delete MS;
  delete P;
  delete EL;
  if (st != TE_OK) return st;
  for (const TcJob& J : jobs) {
    if (!J.e_out) continue;
    ++h->n_launches;
    cudaError_t e = J.t_end > J.t_begin ? launch_reduce_total(J.shares, J.t_end - J.t_begin, J.e_out, s)
                                        : cudaMemsetAsync(J.e_out, 0, sizeof(double), s);
    if (e != cudaSuccess) return fail(TE_ECUDA, "reduction launch: %s", cudaGetErrorString(e));
  }
  return TE_OK;
}

// Plan, buffers (carved from base), operand preparation and maps of one job.
static te_status setup_job(Handle* h, TcState* st, const te_cluster* c, int mode, int64_t t_begin, int64_t t_end,
                           const TcPlan& pl, char* base, TcJob* J, int64_t cluster, cudaStream_t s,
                           const te_df* df = nullptr, const DfScratch* dfs = nullptr) {
  J->c = c;
  J->pl = pl;
  J->o = (int)c->nocc;
  J->v = (int)c->nvir;
  J->t_begin = t_begin;
  J->t_end = t_end;
  J->nbt = energy_num_block_triples(J->v);
  J->slot_floats = g_slot_floats(J->v, pl.fmt);
  J->tiles_per_triple = 3LL * pl.n_mp * pl.n_nt;
  tc_carve_cluster(base, pl, J->o, J->v, num_unique_triples(J->o), &J->b);
  J->shares = J->b.etri;
  te_status rs = launch_prep_tc(h, mode, c, pl, J->b, df, dfs, h->d_err, cluster, s);
  if (rs != TE_OK) return rs;
  rs = build_maps(st, pl, J->o, J->v, J->b, &J->maps);
  if (rs != TE_OK) return rs;
  return build_energy_maps(st, pl, J->o, J->v, J->b, &J->em);
}

static te_status check_k(int mode, int o, int v) {
  // exact level-0/1 sums: K = 2 (v + o) products of at most 2^(2 beta) units stay below 2^24
  if (mode == TC_OZAKI6 && 2 * (v + o) > OZ_K_MAX6)
    return fail(TE_EUNSUPPORTED, "OZAKI mode needs 2 (nvir + nocc) <= %d for exact accumulation", OZ_K_MAX6);
  if (mode == TC_OZAKI && 2 * (v + o) > OZ_K_MAX7)
    return fail(TE_EUNSUPPORTED, "7-bit OZAKI slices need 2 (nvir + nocc) <= %d (use 6-bit slices)", OZ_K_MAX7);
  return TE_OK;
}

static TcPool single_pool(const TcPlan& pl, int v) {
  TcPool q;
  q.pool_floats = (int64_t)pl.nslots * g_slot_floats(v, pl.fmt);
  q.max_slots = pl.nslots;
  q.par_slots = pl.par_slots;
  return q;
}

// The forms of a single-cluster call and their workspace: the usual one, then
// half the triples per launch and again, down to min_slots, with a share
// reduction per launch, where memory is short.  The shares have the same bits.
struct SingleForms {
  std::vector<TcPlan> plan;
  std::vector<size_t> bytes;
};
static SingleForms single_forms(const Handle* h, TcPlan pl, int o, int v, const te_df* df) {
  SingleForms f;
  TcBuffers b;
  DfScratch d;
  const size_t fixed = tc_carve_cluster(nullptr, pl, o, v, num_unique_triples(o), &b);
  const size_t form = df ? df_carve(nullptr, o, v, df->naux, &d) : size_t(0);
  for (;;) {
    f.plan.push_back(pl);
    f.bytes.push_back(fixed + std::max(tc_shared_bytes(single_pool(pl, v), h->num_sms), form));
    if (pl.nslots == pl.min_slots && pl.par_slots == pl.nslots) return f;
    pl.nslots = std::max(pl.min_slots, pl.nslots / 2);
    pl.par_slots = pl.nslots;
  }
}

size_t tc_slices_bytes(int o, int v, int ns) {
  const size_t vp = (size_t)round_up(v, 16), op = (size_t)round_up(o, 16), NS = (size_t)ns, es = 2;
  const size_t na = (size_t)o * v * v * vp, nb = (size_t)o * o * v * vp;
  const size_t nl = (size_t)o * v * v * op, nn = (size_t)o * o * v * op;
  auto al = [](size_t b) { return (b + 1023) & ~size_t(1023); };
  const size_t ng = 2 * (size_t)o + 2 * (size_t)o * o;  // row groups of the four arrays
  return al(NS * na * es) + al(NS * nb * es) + al(NS * nl * es) + al(NS * nn * es) + al(ng * 8) + al(ng * 4) + 1024;
}

te_status tc_prepare_slices(const te_cluster* c, void* base_v, SliceSet* out, int num_sms, cudaStream_t s,
                            int ns, unsigned int* err, int64_t cluster, int64_t* launches) {
  const int o = (int)c->nocc, v = (int)c->nvir;
  const int vp = round_up(v, 16), op = round_up(o, 16);
  if (ns != 4 && ns != 5) return fail(TE_EINVAL, "slice count %d (4 or 5)", ns);
  const int NS = ns;
  const size_t es = 2;
  char* base = reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(base_v) + 1023) & ~uintptr_t(1023));
  size_t off = 0;
  auto take = [&](size_t bytes) {
    off = (off + 1023) & ~size_t(1023);
    char* p = base + off;
    off += bytes;
    return p;
  };
  const size_t na = (size_t)o * v * v * vp, nb = (size_t)o * o * v * vp;
  const size_t nl = (size_t)o * v * v * op, nn = (size_t)o * o * v * op;
  char* A = take(NS * na * es);
  char* B = take(NS * nb * es);
  char* L = take(NS * nl * es);
  char* N = take(NS * nn * es);
  const int64_t oo = (int64_t)o * o, ng = 2 * (int64_t)o + 2 * oo;
  auto* hi = reinterpret_cast<unsigned int*>(take((size_t)ng * 8));  // largest magnitudes, laid out as exps
  int* exps = reinterpret_cast<int*>(take((size_t)ng * 4));
  int* e_ovvv = exps;           // [o]
  int* e_t2 = e_ovvv + o;       // [o o]
  int* e_t2L = e_t2 + oo;       // [o]
  int* e_nooT = e_t2L + o;      // [o o]
  Parts pa{}, pb{}, pL{}, pN{};
  for (int k = 0; k < NS; ++k) {
    pa.p[k] = A + (size_t)k * v * v * vp * es;
    pb.p[k] = B + (size_t)k * v * vp * es;
    pL.p[k] = L + (size_t)k * v * v * op * es;
    pN.p[k] = N + (size_t)k * v * op * es;
  }
  // one scale per row group (each strided GEMM reads one group of each
  // operand), so a block far below the array's largest keeps its 28 bits
  const int64_t v2 = (int64_t)v * v, ov = (int64_t)o * v;
  MaxOut mo{};
  mo.groups = true;
  mo.ovvv = hi;
  mo.t2 = hi + o;
  mo.t2L = hi + o + oo;
  mo.ooov = hi + 2 * o + oo;
  cudaError_t e = cudaMemsetAsync(hi, 0, (size_t)ng * 4, s);
  if (e == cudaSuccess) e = launch_check_inputs(c, cluster, err, num_sms, s, nullptr, &mo);
  const SplitScales sc{nullptr, nullptr, hi, exps, (int)ng};
  const SplitJob jobs[4] = {
      {SPLIT_ROWS, c->ovvv, pa, nullptr, v, vp, o * v2, 1, 0, 0, v2, 1, 0, e_ovvv, 0},
      {SPLIT_ROWS, c->t2, pb, nullptr, v, vp, (int64_t)o * o * v, 1, 0, 0, v, 1, 0, e_t2, 0},
      {SPLIT_COLS, c->t2, pL, nullptr, o, op, v2, o, v2, o * v2, v2, 1, 0, e_t2L, 0},
      {SPLIT_COLS, c->ooov, pN, nullptr, o, op, ov, o, o * ov, ov, v, -1, 0, e_nooT, 0}};
  if (e == cudaSuccess) e = launch_split(NS == 5 ? TC_SLICE5 : TC_SLICE4, jobs, 4, sc, s);
  *launches += 2;
  if (e != cudaSuccess) return fail(TE_ECUDA, "slice preparation launch failed: %s", cudaGetErrorString(e));
  out->ovvv = A;
  out->t2 = B;
  out->t2L = L;
  out->nooT = N;
  out->ovvv_plane = (int64_t)v * v * vp;
  out->t2_plane = (int64_t)v * vp;
  out->t2L_plane = (int64_t)v * v * op;
  out->nooT_plane = (int64_t)v * op;
  out->ovvv_p = NS * (int64_t)v * v * vp;
  out->t2_rq = NS * (int64_t)v * vp;
  out->t2L_q = NS * (int64_t)v * v * op;
  out->nooT_pr = NS * (int64_t)v * op;
  out->vp = vp;
  out->op = op;
  out->ns = NS;
  out->e_ovvv = e_ovvv;
  out->e_t2 = e_t2;
  out->e_t2L = e_t2L;
  out->e_nooT = e_nooT;
  return TE_OK;
}

te_status tc_workspace_bytes(Handle* h, const te_cluster* c, te_precision p, size_t* bytes, const te_df* df) {
  const int o = (int)c->nocc, v = (int)c->nvir;
  const TcPlan pl = make_plan(h, o, v, tc_mode_of(p, o, v, h->ozaki_bits), num_unique_triples(c->nocc));
  for (size_t b : single_forms(h, pl, o, v, df).bytes) {
    *bytes = b;  // the first that the limit admits, else the smallest
    if (!h->ws_limit || b <= h->ws_limit) break;
  }
  return TE_OK;
}

std::vector<size_t> tc_energy_bytes(const Handle* h, int o, int v, te_precision p) {
  return single_forms(h, make_plan(h, o, v, tc_mode_of(p, o, v, h->ozaki_bits), num_unique_triples(o)), o, v, nullptr).bytes;
}

te_status ensure_workspace_public(Handle* h, size_t bytes);
te_status ensure_triples_public(Handle* h, int nocc);

te_status tc_autotune(Handle* h, const te_cluster* c, te_precision p, cudaStream_t s) {
  const int o = (int)c->nocc, v = (int)c->nvir, mode = tc_mode_of(p, o, v, h->ozaki_bits);
  const auto key = std::make_tuple(o, v, mode);
  if (h->tuned.count(key)) return TE_OK;
  if (check_k(mode, o, v) != TE_OK) return TE_OK;  // run_tc reports it
  const int64_t nt = num_unique_triples(o);
  if (nt == 0) return TE_OK;
  // candidate M tiles: padding within 15% of the least; candidate N splits: the fewest and one more
  std::vector<std::pair<int, int>> cand;
  int64_t best_rows = -1;
  for (int TB = 128; TB >= 16; TB /= 2) {
    const int TA = 128 / TB;
    const int64_t rows = (int64_t)round_up(v, TA) * round_up(v, TB);
    if (best_rows < 0 || rows < best_rows) best_rows = rows;
  }
  const TcPlan base = make_plan(h, o, v, mode, nt, 128, 0);
  for (int TB = 128; TB >= 16; TB /= 2) {
    const int TA = 128 / TB;
    const int64_t rows = (int64_t)round_up(v, TA) * round_up(v, TB);
    if (rows * 100 > best_rows * 115) continue;
    cand.emplace_back(TB, base.n_nt);
    // one more N split (smaller N tiles re-read the A operand more often)
    if (round_up((v + base.n_nt) / (base.n_nt + 1), 32) < base.NT) cand.emplace_back(TB, base.n_nt + 1);
  }
  if (cand.size() <= 1) {
    if (!cand.empty()) h->tuned[key] = cand[0];
    return TE_OK;
  }
  const auto cached = h->tune_file.find(key);  // a cache file's pick, if it is one of these
  if (cached != h->tune_file.end() && std::find(cand.begin(), cand.end(), cached->second) != cand.end()) {
    h->tuned[key] = cached->second;
    return TE_OK;
  }
  TcState* st = tc_state(h);
  te_status rs = get_encoder(st);
  if (rs != TE_OK) return rs;
  rs = ensure_triples_public(h, o);
  if (rs != TE_OK) return rs;
  size_t need = 0;
  for (const auto& cd : cand) {
    TcPlan pl = make_plan(h, o, v, mode, nt, cd.first, cd.second);
    pl.nslots = pl.par_slots = pl.min_slots;
    TcBuffers b;
    need = std::max(need, tc_carve_cluster(nullptr, pl, o, v, nt, &b) + tc_shared_bytes(single_pool(pl, v), h->num_sms));
  }
  rs = ensure_workspace_public(h, need);
  if (rs != TE_OK) return rs;
  char* wbase = reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(h->ws) + 1023) & ~uintptr_t(1023));
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess)
    return fail(TE_ECUDA, "event creation failed");
  float best_ms = 1e30f;
  std::pair<int, int> best = cand[0];
  bool prepped = false;
  std::vector<TcJob> jobs(1);
  TcMapSet* MS = new TcMapSet;
  TcParams* P = new TcParams;
  for (const auto& cd : cand) {
    TcPlan pl = make_plan(h, o, v, mode, nt, cd.first, cd.second);
    pl.nslots = pl.par_slots = pl.min_slots;
    if (pl.stages < 2) continue;
    TcJob& J = jobs[0];
    J = TcJob{};
    J.c = c;
    J.pl = pl;
    J.o = o;
    J.v = v;
    J.nbt = energy_num_block_triples(v);
    J.slot_floats = g_slot_floats(v, pl.fmt);
    J.tiles_per_triple = 3LL * pl.n_mp * pl.n_nt;
    const size_t cbytes = tc_carve_cluster(wbase, pl, o, v, nt, &J.b);
    cudaError_t e = cudaSuccess;
    if (!prepped) {  // the operand planes sit first in the workspace for every candidate
      if (launch_prep_tc(h, mode, c, pl, J.b, nullptr, nullptr, nullptr, 0, s) != TE_OK) e = cudaErrorUnknown;
      prepped = true;
    }
    if (e != cudaSuccess || build_maps(st, pl, o, v, J.b, &J.maps) != TE_OK) continue;
    const int ns = (int)std::min<int64_t>(pl.nslots, nt);
    TcPiece pc{};
    pc.cl = 0;
    pc.ns = ns;
    pc.nbt = J.nbt;
    pc.gbuf = reinterpret_cast<float*>(wbase + cbytes);
    const int jl[1] = {0};
    size_t smem = 0;
    if (gemm_params(h, jobs, jl, 1, &pc, 1, (int64_t)ns * J.tiles_per_triple, mode, P, MS, &smem) != TE_OK) continue;
    float ms = 1e30f;
    for (int rep = 0; rep < 2; ++rep) {
      cudaEventRecord(e0, s);
      e = launch_gemm_any(mode, *MS, *P, smem, h->num_sms, s);
      cudaEventRecord(e1, s);
      h->n_launches += 1;
      if (e != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess) break;
      float tms = 0.f;
      cudaEventElapsedTime(&tms, e0, e1);
      ms = std::min(ms, tms / (float)ns);  // per triple
    }
    if (h->log)
      std::fprintf(stderr, "[tenergy] autotune nocc=%d nvir=%d mode=%d: TB=%d n_nt=%d %.4f ms per triple\n", o, v,
                   mode, cd.first, cd.second, (double)ms);
    if (ms < best_ms) {
      best_ms = ms;
      best = cd;
    }
  }
  delete MS;
  delete P;
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (cudaGetLastError() != cudaSuccess) return fail(TE_ECUDA, "autotune launch failed");
  h->tuned[key] = best;
  if (h->log)
    std::fprintf(stderr, "[tenergy] autotune nocc=%d nvir=%d mode=%d: picked TB=%d n_nt=%d\n", o, v, mode,
                 best.first, best.second);
  tune_save(h);
  return TE_OK;
}

te_status run_tc(Handle* h, const te_cluster* c, te_precision p, int64_t t_begin, int64_t t_end,
                 double* e_tri_out, double* e_total_out, cudaStream_t s, const te_df* df) {
  if (h->cc_major != 10 && h->cc_major != 11)
    return fail(TE_EUNSUPPORTED, "tensor-core modes need an sm_100-family GPU (found sm_%d%d)", h->cc_major,
                h->cc_minor);
  TcState* st = tc_state(h);
  te_status rs = get_encoder(st);
  if (rs != TE_OK) return rs;
  const int o = (int)c->nocc, v = (int)c->nvir;
  const int mode = tc_mode_of(p, o, v, h->ozaki_bits);
  const int64_t ntri = num_unique_triples(o);
  TcPlan pl = make_plan(h, o, v, mode, t_end - t_begin);
  if (pl.stages < 2) return fail(TE_EUNSUPPORTED, "not enough shared memory for two pipeline stages");
  rs = check_k(mode, o, v);
  if (rs != TE_OK) return rs;
  const SingleForms forms = single_forms(h, pl, o, v, df);
  size_t form = 0;
  rs = acquire_workspace(h, forms.bytes, &form);
  if (rs != TE_OK) return rs;
  pl = forms.plan[form];
  if (h->log)
    std::fprintf(stderr,
                 "[tenergy] plan nocc=%d nvir=%d mode=%d: M tile %d x %d, N tile %d (%d per row block), %d stages "
                 "of %u bytes, %d triples per launch, %u TMEM columns (%d accumulator sets), workspace %zu bytes\n",
                 o, v, mode, pl.TA, pl.TB, pl.NT, pl.n_nt, pl.stages, pl.stage_bytes, pl.nslots, pl.tmem_cols,
                 pl.nbuf, forms.bytes[form]);
  rs = ensure_triples_public(h, o);
  if (rs != TE_OK) return rs;
  TcBuffers b;
  DfScratch dfs;
  const TcPool pq = single_pool(pl, v);
  const size_t cbytes = tc_carve_cluster(nullptr, pl, o, v, ntri, &b);
  char* base = reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(h->ws) + 1023) & ~uintptr_t(1023));
  std::vector<TcJob> jobs(1);
  if (df) df_carve(base + cbytes, o, v, df->naux, &dfs);  // over the G pool, before its first use
  rs = setup_job(h, st, c, mode, t_begin, t_end, pl, base, &jobs[0], 0, s, df, df ? &dfs : nullptr);
  if (rs != TE_OK) return rs;
  if (e_tri_out) jobs[0].shares = e_tri_out;  // shares[t - t_begin]
  else jobs[0].shares = jobs[0].b.etri;
  jobs[0].e_out = e_total_out;
  float* pool = reinterpret_cast<float*>(base + cbytes);
  double* partials = reinterpret_cast<double*>(base + cbytes + (((size_t)pq.pool_floats * 4 + 1023) & ~size_t(1023)));
  return run_rounds(h, jobs, mode, pool, pq, partials, s);
}

// Batches: every member's operands prepared up front, then rounds that mix
// members (largest first), so the whole batch takes a few launches per round
// instead of three per member per slot group.
static constexpr int64_t BATCH_POOL_BYTES = int64_t(16) << 30;

static TcPool batch_pool(Handle* h, const te_cluster* cs, int64_t n, int mode_p) {
  int64_t need = 0, biggest = 0;
  for (int64_t x = 0; x < n; ++x) {
    const int o = (int)cs[x].nocc, v = (int)cs[x].nvir;
    const int mode = tc_mode_of((te_precision)mode_p, o, v, h->ozaki_bits);
    const int64_t sf = g_slot_floats(v, make_plan(h, o, v, mode, num_unique_triples(o)).fmt);
    need += num_unique_triples(o) * sf;
    biggest = std::max(biggest, sf);
  }
  TcPool q;
  q.pool_floats = std::max(biggest, std::min<int64_t>(need, BATCH_POOL_BYTES / 4));
  q.max_slots = 2048;
  q.par_slots = q.max_slots;
  return q;
}

te_status tc_batched_bytes(Handle* h, const te_cluster* cs, int64_t n, te_precision p, size_t* bytes) {
  size_t b = 0;
  for (int64_t x = 0; x < n; ++x) {
    const int o = (int)cs[x].nocc, v = (int)cs[x].nvir;
    const TcPlan pl = make_plan(h, o, v, tc_mode_of(p, o, v, h->ozaki_bits), num_unique_triples(o));
    TcBuffers bb;
    b += tc_carve_cluster(nullptr, pl, o, v, num_unique_triples(o), &bb);
  }
  *bytes = b + tc_shared_bytes(batch_pool(h, cs, n, (int)p), h->num_sms) + 1024;
  return TE_OK;
}

te_status run_tc_batched(Handle* h, const te_cluster* cs, int64_t n, te_precision p, double* e_out, cudaStream_t s) {
  if (h->cc_major != 10 && h->cc_major != 11)
    return fail(TE_EUNSUPPORTED, "tensor-core modes need an sm_100-family GPU (found sm_%d%d)", h->cc_major,
                h->cc_minor);
  TcState* st = tc_state(h);
  te_status rs = get_encoder(st);
  if (rs != TE_OK) return rs;
  size_t bytes = 0;
  tc_batched_bytes(h, cs, n, p, &bytes);
  rs = ensure_workspace_public(h, bytes);
  if (rs != TE_OK) return rs;
  char* base = reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(h->ws) + 1023) & ~uintptr_t(1023));
  // longest first: the rounds' last pieces are the small members
  std::vector<int64_t> order(n);
  for (int64_t x = 0; x < n; ++x) order[x] = x;
  std::stable_sort(order.begin(), order.end(), [&](int64_t a, int64_t b) {
    const double fa = (double)num_unique_triples(cs[a].nocc) * cs[a].nvir * cs[a].nvir * cs[a].nvir * (cs[a].nvir + cs[a].nocc);
    const double fb = (double)num_unique_triples(cs[b].nocc) * cs[b].nvir * cs[b].nvir * cs[b].nvir * (cs[b].nvir + cs[b].nocc);
    return fa > fb;
  });
  std::vector<TcJob> jobs;
  std::vector<int> modes;
  jobs.reserve(n);
  size_t off = 0;
  for (int64_t x : order) {
    const int o = (int)cs[x].nocc, v = (int)cs[x].nvir;
    const int mode = tc_mode_of(p, o, v, h->ozaki_bits);
    rs = check_k(mode, o, v);
    if (rs != TE_OK) return rs;
    const int64_t nt = num_unique_triples(o);
    if (nt == 0) {  // no triples: the value checks alone
      if (launch_check_inputs(cs + x, x, h->d_err, h->num_sms, s) != cudaSuccess ||
          cudaMemsetAsync(e_out + x, 0, sizeof(double), s) != cudaSuccess)
        return fail(TE_ECUDA, "check or memset launch failed");
      h->n_launches += 2;
      continue;
    }
    const TcPlan pl = make_plan(h, o, v, mode, nt);
    TcJob J;
    rs = setup_job(h, st, cs + x, mode, 0, nt, pl, base + off, &J, x, s);
    if (rs != TE_OK) return rs;
    TcBuffers bb;
    off += tc_carve_cluster(nullptr, pl, o, v, nt, &bb);
    J.e_out = e_out + x;
    jobs.push_back(J);
    modes.push_back(mode);
  }
  const TcPool pq = batch_pool(h, cs, n, (int)p);
  float* pool = reinterpret_cast<float*>(base + off);
  double* partials = reinterpret_cast<double*>(base + off + (((size_t)pq.pool_floats * 4 + 1023) & ~size_t(1023)));
  // one kernel per mode: the members of each slice width run in their own rounds
  for (int mode : {TC_TF32, TC_BF16X3, TC_TF32X3, TC_OZAKI, TC_OZAKI6}) {
    std::vector<TcJob> group;
    for (size_t q = 0; q < jobs.size(); ++q)
      if (modes[q] == mode) group.push_back(jobs[q]);
    if (group.empty()) continue;
    rs = run_rounds(h, group, mode, pool, pq, partials, s);
    if (rs != TE_OK) return rs;
  }
  return TE_OK;
}

}  // namespace te
