"""The tile of a float64 contraction fits its launch: the SM with the most blocks
has no more float64 work than with tiles of 64 x 64, whatever the output, the
number of products in the launch and the length of K."""
import os
import shutil
import subprocess

import pytest

import paper_2412_18553_gb300

CSRC = os.path.join(os.path.dirname(paper_2412_18553_gb300.__file__), "csrc")
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

PROGRAM = r"""
#include <cstdio>
#include "dfma_tile.cuh"
using namespace te;
int main() {
  const long long cases[][5] = {  // M, N, K, products, doubles of scratch
      CASES};
  for (const auto& c : cases) {
    const DfmaPick t = dfma_pick(c[0], c[1], c[2], c[3], 152, c[4], false);
    std::printf("%d %d %lld %lld %d\n", t.rm, t.nb, (long long)t.tiles_m, (long long)t.tiles_n, t.nsplit);
  }
}
"""


def busiest(tiles, nsplit, products, work, K):
    """Thread-tile elements times k on the busiest of 152 SMs."""
    return -(-tiles * nsplit * products // 152) * work * -(-K // nsplit)


@pytest.mark.skipif(not os.path.exists(NVCC), reason="needs nvcc")
def test_no_sm_has_more_work_than_with_64_by_64_tiles(tmp_path):
    cases = [(v * v, v, K, n, 0) for v in (1, 7, 8, 31, 33, 40, 41, 48, 53, 64, 65, 96, 97, 120)
             for K in (3, 8, v) for n in (1, 3, 24, 700)]
    cases += [(v, o, v * v, 1, 80 * v * v) for o in (1, 4, 8, 14) for v in (8, 37, 48, 96, 120)]
    cases += [(o * v, o * v, 4 * (o + v), 1, 0) for o, v in ((2, 10), (4, 32), (8, 64), (20, 160))]
    src = tmp_path / "pick.cu"
    src.write_text(PROGRAM.replace("CASES", ", ".join("{%d, %d, %d, %d, %d}" % c for c in cases)))
    exe = str(tmp_path / "pick")
    subprocess.run([NVCC, "-std=c++17", "-I", CSRC, str(src), "-o", exe], check=True, capture_output=True, text=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split("\n")
    for (M, N, K, n, cap), line in zip(cases, out):
        rm, nb, tm, tn, ns = (int(x) for x in line.split())
        assert tm * 32 * rm >= M and tn * 8 * nb >= N and ns >= 1 and (ns == 1 or ns * M * N <= cap)
        wide = -(-M // 64) * -(-N // 64)
        steps = -(-K // 16)
        wide_ns = max(1, min(-(-304 // wide), steps // 8, cap // (M * N)))
        # a little more work may buy fewer chunks to stage or partials to add
        assert busiest(tm * tn, ns, n, rm * nb, K) <= 1.1 * busiest(wide, wide_ns, n, 16, K) + 16, (M, N, K, n, line)
