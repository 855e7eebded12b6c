// The inner product of a float64 tile on the DFMA units, shared by the W~
// contraction (gemm_fp64.cu) and the strided-view contractions (vjp.cu).
//
// A block of 256 threads owns 32 RM rows by 8 NB columns; thread (ty, tx) =
// (tid / 8, tid % 8) holds rows ty + 32 a and columns tx + 8 b.  GB300 issues
// two DFMA lanes per SM and cycle, so a warp's DFMA takes 16 cycles of the SM
// against 2 for an 8-byte shared-memory load: even a 1 x 1 thread tile keeps
// the float64 units busy, and what costs time is work on padding.  The tile is
// therefore chosen per launch with the least padded rows and columns
// (dfma_pick); a 64 x 64 tile spent 1.6 times the needed work on 40 columns and
// ten times on a 20 x 20 output.  K is not padded: the last chunk runs its own
// length.
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
};

// The tile with the least padded work for an M x N output: rm in {1, 2, 4},
// nb in 1 .. 8; the larger tile on a tie (fewer loads of the operands).
inline DfmaPick dfma_pick(int64_t M, int64_t N) {
  DfmaPick best{4, 8, 1, 1};
  int64_t cost = -1;
  for (int rm = 4; rm >= 1; rm >>= 1)
    for (int nb = 8; nb >= 1; --nb) {
      const int64_t tm = (M + 32 * rm - 1) / (32 * rm), tn = (N + 8 * nb - 1) / (8 * nb);
      const int64_t c = tm * rm * tn * nb;
      if (cost < 0 || c < cost) {
        cost = c;
        best = DfmaPick{rm, nb, tm, tn};
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
