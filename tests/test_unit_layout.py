"""Shared memory of the fp32 one-kernel runs (host arithmetic of lola_unit_f32.cuh, compiled here without a GPU)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2505_23666_b200", "csrc")

PROBE = r"""
#include <cstdio>
#include <cstdlib>
#include "lola_unit_f32.cuh"
using namespace lola;
int main(int argc, char** argv) {
  for (int i = 1; i + 5 < argc; i += 6) {              // d F K C lambda query-rows -> fits, both groups attend, apart
    const int d = atoi(argv[i]), F = atoi(argv[i + 1]), K = atoi(argv[i + 2]), C = atoi(argv[i + 3]), lam = atoi(argv[i + 4]);
    Layer L{};
    L.d = d; L.F = F; L.D = 2 * F; L.lam = lam; L.cmax = C; L.eta = C;
    const UnitLayout Y = unit_layout(L, K, atoi(argv[i + 5]));
    const int nE = lam + C;
    // what is in use at the same time lies apart, and the scratch of the selection clear of the one value row that is there beside it
    struct { int at, n; } live[] = {{Y.W, d * Y.fp}, {Y.H, Y.dp * d}, {Y.s, Y.dp}, {Y.phi, (nE + K - 1) / K * Y.phi_ld}, {Y.key, nE}, {Y.pos, nE}, {Y.fold, C},
                                    {Y.dst, C}, {Y.src, kUnSrcFloats}, {Y.vf, d}, {Y.sel, (int)sizeof(SelectScratch) / 4}, {Y.cand, nE}, {Y.mark, (nE + 3) / 4}};
    const int n = (int)(sizeof(live) / sizeof(live[0]));
    bool apart = (Y.sel & 3) == 0 && (Y.key & 3) == 0 && Y.sel + (int)sizeof(SelectScratch) / 4 <= Y.pf;
    // the query scratch of a group (the key groups' sums over z and p), a scoring tile and, where it attends too, another set beside it
    const int sets = Y.both ? 2 : 1, set = 8 * d + Y.dp * 8 + 2 * 8 * kUnKeys + 2 * kUnKeys + 24, tile = kUnRows * (d + 4) + kUnRows;
    apart = apart && Y.att0 >= set && Y.row + 24 <= Y.q + Y.att0 && Y.q + sets * Y.att0 <= Y.key && Y.red >= Y.z && Y.red + 4096 <= Y.vptr &&
            Y.xs == Y.q + Y.att0 && Y.den == Y.xs + kUnRows * (d + 4) && Y.xs + tile <= Y.key;
    for (int x = 0; x < n; ++x) {
      apart = apart && live[x].at >= 0 && live[x].at + live[x].n <= Y.total;
      for (int y = 0; y < x; ++y) apart = apart && (live[x].at + live[x].n <= live[y].at || live[y].at + live[y].n <= live[x].at);
    }
    printf("%d %d %d\n", Y.total * 4 <= kUnSmem ? 1 : 0, Y.both, apart ? 1 : 0);
  }
  return 0;
}
"""

SIDE, BOTH = 0, 1
# d, F, blocks per unit, chunk, sparse cache, query rows, how the groups share the work: caches that a block has to hold, up to the largest
HELD = [(64, 64, 8, 16, 1648, 32, SIDE), (64, 64, 8, 32, 1620, 64, SIDE), (64, 64, 8, 64, 1556, 512, SIDE), (64, 64, 8, 64, 1728, 64, SIDE),
        (64, 64, 8, 100, 1488, 100, SIDE), (64, 64, 1, 64, 160, 64, SIDE), (64, 64, 4, 512, 384, 512, SIDE),
        (64, 65, 1, 64, 160, 64, SIDE), (64, 65, 1, 16, 208, 16, SIDE), (64, 32, 8, 64, 3348, 64, SIDE), (64, 1, 4, 64, 9024, 64, SIDE),
        (64, 1, 8, 64, 11156, 64, SIDE), (64, 16, 2, 64, 2048, 64, SIDE),
        (128, 64, 8, 64, 704, 64, SIDE), (128, 64, 8, 64, 704, 65, BOTH), (128, 64, 8, 64, 960, 512, BOTH), (128, 64, 8, 64, 960, 0, SIDE),
        (128, 65, 8, 64, 704, 128, BOTH), (128, 65, 8, 64, 832, 128, SIDE), (128, 65, 8, 64, 960, 64, SIDE),
        (128, 64, 4, 64, 448, 64, BOTH), (128, 64, 4, 64, 448, 32, SIDE), (128, 64, 2, 64, 192, 64, BOTH), (128, 64, 1, 64, 32, 64, BOTH),
        (128, 64, 1, 64, 32, 8, SIDE), (128, 32, 1, 64, 384, 64, BOTH), (128, 32, 2, 512, 384, 512, BOTH), (128, 16, 1, 64, 960, 64, BOTH),
        (128, 65, 2, 128, 128, 128, BOTH), (128, 65, 2, 256, 0, 256, BOTH), (128, 1, 8, 64, 10920, 64, SIDE)]


@pytest.fixture(scope="module")
def layouts(tmp_path_factory):
    from paper_2505_23666_b200.build import _nvcc
    tmp = tmp_path_factory.mktemp("layout")
    src, exe = tmp / "probe.cu", tmp / "probe"
    src.write_text(PROBE)
    subprocess.run([_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-w", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    args = [str(x) for case in HELD for x in case[:6]]
    return [tuple(map(int, line.split())) for line in subprocess.run([str(exe)] + args, check=True, capture_output=True, text=True).stdout.splitlines()]


@pytest.mark.parametrize("i", range(len(HELD)), ids=[str(c) for c in HELD])
def test_sparse_caches_that_one_block_holds(layouts, i):
    fits, both, apart = layouts[i]
    assert fits == 1 and apart == 1 and both == HELD[i][6]
