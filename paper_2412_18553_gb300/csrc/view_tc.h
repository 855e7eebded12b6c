// Exact-slice contractions on tcgen05 over tensor-map views (view_tc.cu).
//
// One launch runs a list of jobs.  A job is an output C[(m1, m2), n] in
// float64 and a list of K segments, each
//   C[(m1, m2), n] += alpha 2^(ea + eb) sum_{k1, k2} A[(m1, m2), (k1, k2)] B[n, (k1, k2)]
// (alpha = +-1 per segment)
// where A and B are BF16 slice planes (value = 2^e sum_s slice_s) read through
// TMA tensor maps whose innermost dimension is the contiguous K index k2.
// Slice products a_i b_j with i + j <= NS - 1 go to three FP32 accumulators in
// tensor memory (level 0, level 1, the rest); K is taken in blocks of at most
// 1024 elements, so the level-0 and level-1 sums are exact.  A unit adds its
// blocks in double-float (FP32 pairs, 2^-48 relative) and its total to C (or
// to a split-K partial) in float64.
//
// Work unit: (job, m tile or pair of m tiles, n tile, K split).  A unit owns its
// output tile (or its split's partial tile) for the whole launch, so no two
// units write the same element and the result has a fixed summation order.
// Jobs of one launch must write disjoint outputs.
//
// A launch runs on pairs of CTAs (cta_group::2: two m tiles against one B tile of
// which each CTA holds half) or on lone CTAs, for jobs whose rows fill one
// tile only.  The B maps of a pair launch have boxes of NT / 2 rows, those of a
// lone launch NT rows.
#pragma once
#include <cuda.h>

#include <cstdint>

#include "te_internal.h"

namespace te {

constexpr int VT_MAX_MAPS = 20;
constexpr int VT_MAX_SEGS = 288;     // per launch: the tables travel as kernel parameters (32 KB)
constexpr int VT_MAX_JOBS = 96;
constexpr int VT_KC = 32;            // K elements per pipeline stage: 64-byte rows, 64-byte swizzle
constexpr int VT_BLOCK_CHUNKS = 32;  // stages per exact accumulation block: K <= 1024
constexpr int VT_NT_MAX = 128;       // N tile: three accumulators; an epilogue thread holds NT/2 column sums
constexpr int VT_NT_PAIR = 64;       // the same on CTA pairs

// Which of a tensor map's five dimensions holds each index of the view; -1 when
// the view has no such index (r1 for single-index rows, k1 when K = k2 alone).
// k2 is always dimension 0 (contiguous); rows r2 come before r1 and before the
// slices s, which one copy brings together.  rows: the box's row count.
struct VtRoles {
  int8_t k2, r2, r1, k1, s;
  int16_t rows;
};

struct VtSeg {
  int8_t amap, bmap;
  int16_t sign;              // +1 or -1
  int16_t afix[3], bfix[3];  // coordinates of dimensions 2, 3, 4 where they have no role (group indices)
  int nk2c;                  // stages along k2: ceil(K2 / VT_KC)
  int nchunks;               // K1 * nk2c
  const int* ea;             // scale exponents (device)
  const int* eb;
};

// float64 +=, float64 =, or the unit's FP32 pair (hi, lo), |lo| <= ulp(hi) / 2,
// relative to 2^(the largest scale of the job's segments).  One kind per launch; VT_PAIR on CTA pairs only.  VT_ADD (and VT_STORE on lone CTAs) sums a unit's blocks to 2^-48 of the sum;
// VT_STORE on pairs and VT_PAIR round the higher levels' part to FP32 against the low
// word first (2^-38 of the operands' scale; few blocks per unit).  VT_STORE is the
// adjoint's G, whose last bits decide how dW~ is cut.
enum VtOut { VT_ADD = 0, VT_STORE = 1, VT_PAIR = 2 };

struct VtJob {
  int M1, M2, N;
  int16_t TA, TB, NT;  // row tile TA values of m1 x TB values of m2 (TA TB = 128); NT columns
  int16_t out;         // VtOut; VT_STORE and VT_PAIR run unsplit
  int16_t seg0, nseg;  // segments in VtParams::seg
  int16_t bchunks;     // stages per accumulation block
  int16_t vec;         // four columns per access (contiguous, 32-byte aligned)
  int nm2, nmu, nn, nsplit;  // m tiles along m2, units along m, N tiles
  int64_t unit0;       // first unit of the job in the launch
  int64_t nblocks;     // accumulation blocks over all segments
  void* C;             // element (m1, m2, n) at m1 c_m1 + m2 c_m2 + n c_n
  int64_t c_m1, c_m2, c_n;
  double* part;        // nsplit > 1: [nsplit][M1 M2][N], added into C by vt_launch
  int64_t red0;        // first element of the job in the launch's split-reduction index space
};

struct VtMaps {
  CUtensorMap m[VT_MAX_MAPS];
};

struct VtParams {
  int njobs, ns, nsegs;
  int stages;
  uint32_t stage_bytes;  // A part (ns x 128 rows x 64 B) then B part (ns x nt_max rows x 64 B)
  uint32_t tmem_cols;
  int nt_max;
  int64_t total_units;
  int64_t total_red;     // outputs of the split jobs
  unsigned int* err;
  unsigned long long wait_ns;
  VtRoles roles[VT_MAX_MAPS];
  VtJob job[VT_MAX_JOBS];
  VtSeg seg[VT_MAX_SEGS];
};
static_assert(sizeof(VtMaps) + sizeof(VtParams) <= 32764, "kernel parameters");

// A BF16 slice array seen through a five-dimensional tensor map: dims and
// strides in elements (stride[0] = 1), the roles of the dimensions, and the
// plane stride is the stride of the role-s dimension.
struct VtView {
  const void* base;
  uint64_t dims[5];
  uint64_t stride[5];
  VtRoles roles;
};

// Encoded views shared by the launches of one call.
constexpr int VT_BANK_MAX = 24;
struct VtBank {
  CUtensorMap m[VT_BANK_MAX];
  VtRoles r[VT_BANK_MAX];
  int n;
};
// Encode a view (rows per box: rows_r2 x rows_r1, rows_r1 = 1 for
// single-index rows; all ns slices) as bank entry *idx; fails if a stride or the
// base breaks the tensor-map rules.
te_status vt_bank_add(VtBank* k, const VtView& v, int rows_r2, int rows_r1, int* idx);

// Host-side launch under construction.
struct VtBuild {
  VtMaps maps;
  VtParams P;
  int nmaps;
  int8_t slot[VT_BANK_MAX];  // launch-local map index of each bank entry, -1 if unused
  bool pair, full;           // full: a table overflowed
};

// pair: run on CTA pairs
void vt_begin(VtBuild* b, int ns, bool pair);
// launch-local map index of bank entry idx (copied on first use); -1 when the
// launch holds VT_MAX_MAPS maps already
int vt_use(VtBuild* b, const VtBank& k, int idx);
// Append a job (null when the launch is full; vt_finish reports it); its
// segments follow by vt_seg before the next job.
VtJob* vt_job(VtBuild* b, int M1, int M2, int N, int TA, int TB, int NT, void* C, int64_t c_m1, int64_t c_m2,
              int64_t c_n, VtOut out);
// afix, bfix: coordinates of dimensions 2, 3, 4
void vt_seg(VtBuild* b, int amap, int bmap, int K1, int K2, const int* afix, const int* bfix, const int* ea,
            const int* eb, int sign);
// Choose split counts (jobs that overwrite, or all jobs when part_scratch is
// null, keep one split) and unit offsets; part_scratch holds the partials,
// consecutively per split job.  The doubles of scratch used go to *used.
te_status vt_finish(VtBuild* b, int num_sms, double* part_scratch, int64_t scratch_cap, int64_t* used);
// Split count and partial doubles vt_finish chooses for a job of `tiles`
// output tiles, `nblocks` accumulation blocks and mn outputs.
int64_t vt_splits(int64_t tiles, int64_t nblocks, int units_at_once);
int64_t vt_split_doubles(int64_t tiles, int64_t nblocks, int64_t mn, int units_at_once);
// Accumulation blocks of one segment over K = K1 x K2 with bchunks stages per
// block.
int64_t vt_seg_blocks(int K1, int K2, int bchunks = VT_BLOCK_CHUNKS);
// Stages per block for a job with few output tiles (more units to split K
// over; each block still ends in exact level-0/1 sums).
constexpr int VT_SPLIT_CHUNKS = 8;
// Launch the units (grid: min(units, SMs)), then add the split partials of
// every job into C in split order.
te_status vt_launch(Handle* h, VtBuild* b, cudaStream_t s);

// N tile for an output of n columns: at most VT_NT_MAX in steps of 16, on CTA pairs
// VT_NT_PAIR in steps of 32.
int vt_ntile(int64_t n, bool pair);

// C[i][j] = 2^(ea + eb) sum_k A[i][k] B[j][k] (i < m, j < n; C has rows of n) over ns
// slice planes with rows of Kp elements (Kp a multiple of 8, planes 16-byte aligned),
// on lone CTAs.  K is taken in blocks of VT_PRODUCT_CHUNKS stages: the third
// accumulator cuts what every MMA adds at 2^-24 of its sum, and where the slices'
// products have one sign (the diagonal of (ia|jb)) that error grows with the square
// of a block's length: 1.7e-9 of the scale's square at K = 1024 in blocks of 128,
// 2.4e-8 in one block.  The ovvv of nocc=16 nvir=160 from 704 auxiliary functions
// (five slices): 1.84 ms, 1.17 in one block, 3.40 with mma.sync on row-contiguous
// factors.
constexpr int VT_PRODUCT_CHUNKS = 4;
te_status vt_product(Handle* h, const void* a, int64_t a_plane, int64_t m, const void* b, int64_t b_plane, int64_t n,
                     int64_t K, int64_t Kp, int ns, const int* ea, const int* eb, double* C, cudaStream_t s);

struct SliceSet;
// The six views of an exact-slice operand set (tc_prepare_slices) that the
// four K segments of a G block read, rows (x, y) in tiles of 8 x 16 and z in
// tiles of nt (pair launches): idx[0..5] = ovvv rows (x, y), ovvv rows (y, x), t2L rows
// (x, y), t2L rows (y, x), t2 rows z, nooT rows z.  Group coordinates: ovvv
// and t2L take their occupied index at dimension 4; t2[r][q] takes q at 3 and
// r at 4; nooT[p][r] takes r at 3 and p at 4.
te_status vt_slice_maps(VtBank* k, const SliceSet& S, int o, int v, int nt, int* idx);

// Tiled transpose of BF16 slice planes: for every plane p < np and batch b <
// nb, dst[p][b][c][r] = src[p][b][r][c] over r < R, c < Cc (element strides
// given; the innermost index of each side is contiguous).
cudaError_t vt_transpose(const void* src, int64_t src_ps, int64_t src_bs, int64_t src_rs, void* dst,
                         int64_t dst_ps, int64_t dst_bs, int64_t dst_cs, int np, int nb, int R, int Cc,
                         cudaStream_t s);

}  // namespace te
