// The inner product of a float64 tile on the DFMA units, shared by the W~
// contraction (gemm_fp64.cu) and the strided-view contractions (vjp.cu).
//
// A block of 256 threads owns 32 RM rows by 8 NB columns; thread (ty, tx) =
// (tid / 8, tid % 8) holds rows ty + 32 a and columns tx + 8 b.  GB300 issues
// two DFMA lanes per SM and cycle, so a warp's DFMA takes 16 cycles of the SM
// against 2 for an 8-byte shared-memory load: even a 1 x 1 thread tile keeps
// the float64 units busy, and what costs time is work on padding and SMs without
// any.  The tile is therefore chosen per launch (dfma_pick); a 64 x 64 tile spent
// 1.6 times the needed work on 40 columns and ten times on a 20 x 20 output, and
// the least padding alone put one 2304 x 48 product on 18 of 152 SMs.  K is not
// padded: the last chunk runs its own length.
#pragma once
#include <cstdint>
#include <type_traits>

namespace te {

constexpr int DT_K = 16;        // K chunk
constexpr int DT_THREADS = 256;

template <int RM, int NB>
struct DfmaSmem {
  double a[DT_K][32 * RM + 1];
  double b[DT_K][8 * NB + 1];
};

template <int RM, int NB>
__device__ __forceinline__ void dfma_one(const DfmaSmem<RM, NB>& S, int kk, int tx, int ty, double (&acc)[RM][NB]) {
  double av[RM], bv[NB];
#pragma unroll
  for (int a = 0; a < RM; ++a) av[a] = S.a[kk][ty + 32 * a];
#pragma unroll
  for (int b = 0; b < NB; ++b) bv[b] = S.b[kk][tx + 8 * b];
#pragma unroll
  for (int a = 0; a < RM; ++a)
#pragma unroll
    for (int b = 0; b < NB; ++b) acc[a][b] = fma(av[a], bv[b], acc[a][b]);
}

// acc += A[:, 0..kn) B[:, 0..kn)^T of the staged chunk, kk in order
template <int RM, int NB>
__device__ __forceinline__ void dfma_chunk(const DfmaSmem<RM, NB>& S, int kn, double (&acc)[RM][NB]) {
  const int tx = threadIdx.x & 7, ty = threadIdx.x >> 3;
  if (kn >= DT_K) {
#pragma unroll 4
    for (int kk = 0; kk < DT_K; ++kk) dfma_one<RM, NB>(S, kk, tx, ty, acc);
  } else {
    for (int kk = 0; kk < kn; ++kk) dfma_one<RM, NB>(S, kk, tx, ty, acc);
  }
}

struct DfmaPick {
  int rm, nb;
  int64_t tiles_m, tiles_n;
  int nsplit;
};

// Split count for `tiles` output tiles: about two blocks per SM, each split at
// least 8 K chunks, the partial tiles within `cap` doubles.
inline int dfma_splits(int64_t tiles, int64_t K, int64_t MN, int num_sms, int64_t cap) {
  const int64_t steps = (K + DT_K - 1) / DT_K;
  int64_t want = (2LL * num_sms + tiles - 1) / tiles;
  if (want > steps / 8) want = steps / 8;
  if (want > cap / (MN > 0 ? MN : 1)) want = cap / (MN > 0 ? MN : 1);
  return (int)(want > 1 ? want : 1);
}

// The tile (rm in {1, 2, 4}, nb in 1 .. 8) and split count for `copies` products
// M x N over K in one launch, by the time of the SM with the most blocks: 128
// cycles per k for a thread tile of one (8 warps, 16 cycles a DFMA), some for the
// staging of a chunk (which the other blocks of a long queue hide), and the pass
// that adds the splits' partials.  `half`: only the tiles at or below the
// diagonal run.  The larger tile on a tie.
// Eight products of 2304 x 48 over 48 or 8 per G block (the projected energy of
// nocc=8 nvir=48): 177 ms by least padding alone, 47 ms so, 129 ms with 64 x 64 tiles.
inline DfmaPick dfma_pick(int64_t M, int64_t N, int64_t K, int64_t copies, int num_sms, int64_t cap, bool half) {
  DfmaPick best{4, 8, 1, 1, 1};
  int64_t cost = -1;
  for (int rm = 4; rm >= 1; rm >>= 1)
    for (int nb = 8; nb >= 1; --nb) {
      const int64_t tm = (M + 32 * rm - 1) / (32 * rm), tn = (N + 8 * nb - 1) / (8 * nb), tiles = tm * tn;
      const int64_t ns = dfma_splits(tiles, K, M * N, num_sms, cap);
      const int64_t run = half && ns == 1 ? (tiles + (tm > tn ? tm : tn)) / 2 : tiles;
      const int64_t waves = (run * ns * copies + num_sms - 1) / num_sms;
      const int64_t kper = (K + ns - 1) / ns, chunks = (kper + DT_K - 1) / DT_K;
      int64_t c = waves * 128 * rm * nb * kper + (waves < 2 ? waves : 2) * chunks * (64 * rm + 16 * nb + 200);
      if (ns > 1) c += 6000 + M * N * ns / 200;
      if (cost < 0 || c < cost) {
        cost = c;
        best = DfmaPick{rm, nb, tm, tn, (int)ns};
      }
    }
  return best;
}

// f(rm, nb) as integral constants, for the picked tile
template <int RM, typename F>
inline void dfma_dispatch_nb(int nb, F&& f) {
  const std::integral_constant<int, RM> rm;
  switch (nb) {
    case 1: f(rm, std::integral_constant<int, 1>{}); break;
    case 2: f(rm, std::integral_constant<int, 2>{}); break;
    case 3: f(rm, std::integral_constant<int, 3>{}); break;
    case 4: f(rm, std::integral_constant<int, 4>{}); break;
    case 5: f(rm, std::integral_constant<int, 5>{}); break;
    case 6: f(rm, std::integral_constant<int, 6>{}); break;
    case 7: f(rm, std::integral_constant<int, 7>{}); break;
    default: f(rm, std::integral_constant<int, 8>{}); break;
  }
}
template <typename F>
inline void dfma_dispatch(const DfmaPick& p, F&& f) {
  if (p.rm == 1) dfma_dispatch_nb<1>(p.nb, f);
  else if (p.rm == 2) dfma_dispatch_nb<2>(p.nb, f);
  else dfma_dispatch_nb<4>(p.nb, f);
}

}  // namespace te
