// Operand preparation of the tensor-core modes (prep_tc.cu): the largest
// magnitudes that set the scales, and the split of the float64 inputs into
// the parts (hi / lo, or exact slices) that the contractions read.
#pragma once
#include <cuda_bf16.h>

#include "te_internal.h"

namespace te {

// TC_OZAKI: four 7-bit slices, ten slice products (K = 2 (v + o) <= 1024).
// TC_OZAKI6: five 6-bit slices, fifteen slice products (K <= 4096); chosen
// for the same user mode when the K axis is too long for 7-bit slices.
// TC_SLICE4, TC_SLICE5: four or five 7-bit slices, the operand form of the
// view GEMM (no contraction kernel of their own), cut from the integer
// N = round(x 2^(7 NS - s)) in balanced base-128 digits.
enum TcMode { TC_TF32 = 0, TC_BF16X3 = 1, TC_TF32X3 = 2, TC_OZAKI = 3, TC_OZAKI6 = 4, TC_SLICE5 = 5, TC_SLICE4 = 6 };

__host__ __device__ constexpr bool is_ozaki(int mode) {
  return mode == TC_OZAKI || mode == TC_OZAKI6 || mode == TC_SLICE5 || mode == TC_SLICE4;
}

template <int MODE>
struct ModeTraits {
  static constexpr bool tf32 = (MODE == TC_TF32 || MODE == TC_TF32X3);
  static constexpr int nparts =
      (MODE == TC_TF32) ? 1
                        : ((MODE == TC_OZAKI || MODE == TC_SLICE4) ? 4 : ((MODE == TC_OZAKI6 || MODE == TC_SLICE5) ? 5 : 2));
  static constexpr int nacc = is_ozaki(MODE) ? 3 : 1;     // accumulators per tile
  static constexpr int beta = MODE == TC_OZAKI6 ? 6 : 7;  // bits per slice
  static constexpr int es = tf32 ? 4 : 2;                 // bytes per stored element
};

constexpr int MAX_PARTS = 5;

struct Parts {
  void* p[MAX_PARTS];
};

// One piece of the split work of a launch.
//  rows:  dst[row][kp] = src[row][k] (k < K), zero for K <= kp < Kp; `n` rows.
//  cols:  dst[b n + i][l] = sign src[b bs + l ls + i] (l < K), zero for
//         K <= l < Kp; i < n, b < nb: a transpose of l against i.
// Both write slice-interleaved planes: rows come in groups of G (one occupied
// index, or one occupied pair), and a group's parts are consecutive blocks,
// [group][part][G rows][Kp]; parts.p[s] points at part s of group 0.
// The scale exponent of a row is gexp[row / G] when gexp is set, else that of
// entry `which` of SplitExps (exact-slice modes; the others do not scale).
//  ovs:   dst32[i][a][j][b] = 1/2 (src[i,a,j,b] + src[j,b,i,a]), b padded to Kp
//  copy:  dst32[row][kp] = src[row][k], float32
enum SplitKind { SPLIT_ROWS = 0, SPLIT_COLS = 1, SPLIT_OVS = 2, SPLIT_COPY = 3 };
struct SplitJob {
  int kind;
  const double* src;
  Parts parts;
  float* dst32;
  int K, Kp;
  int64_t n, nb, bs, ls, G;
  int sign;  // +1 or -1 (cols)
  int which;
  const int* gexp;
  int64_t block0;  // first block of the job (set by the launch)
};
constexpr int SPLIT_MAX_JOBS = 6;

// Scales of the exact-slice energy modes: one per array, from the high words
// of max |ovvv|, |t2|, |ooov| (maxhi[0..2]), with one unit 2^U for every
// segment of the K axis.  The launch writes {s_ovvv, s_t2, s_t2L, s_nooT, U}
// to exps.  maxhi null: no array scales.
// groups (the SLICE modes): exps[g] of `ngroups` row groups from the high
// words of their largest magnitudes; each job's gexp points into exps, whose
// values the job reads from hi + (gexp - exps) so that one launch does both.
struct SplitScales {
  const unsigned int* maxhi;
  int* exps;
  const unsigned int* group_hi;
  int* group_exps;
  int ngroups;
};

cudaError_t launch_split(int mode, const SplitJob* jobs, int njobs, const SplitScales& sc, cudaStream_t s);

// The largest magnitude of arrays, as the high 32 bits of the float64 (they
// order as integers), and the check that every entry is finite.
struct MaxArray {
  const double* p;
  int64_t rows, len;  // rows of len contiguous entries
  int o;              // group of a row: 0: 0; -1: the row; o > 0: (row / o^2) o + row % o
  unsigned int* out;  // [groups], null: finite check only
  unsigned int* out2; // nullable: a second grouping, group row % o2
  int o2;
  unsigned int site;  // reported (with the cluster) when an entry is not finite; 0: no report
};
constexpr int MAX_ARRAYS = 9;
// eps_o / eps_v (nullable): also check max(eps_o) < min(eps_v) (site 8).  The
// outputs start at zero (the caller clears them).
cudaError_t launch_absmax(const MaxArray* arrays, int n, const double* eps_o, int o, const double* eps_v, int v,
                          unsigned int cluster, unsigned int* err, int num_sms, cudaStream_t s);

}  // namespace te
