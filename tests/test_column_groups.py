"""Which block streams which surviving column in k_spmspv_direct, evaluated by the library's own rules: a group's ranking lanes
hold every column once, every survivor has one taker, no block takes more than its tables hold, and the busiest block has
little more than the mean.  No GPU needed."""
import os
import subprocess

import numpy as np
import pytest

from conftest import ROOT


@pytest.fixture(scope="module")
def takers(tmp_path_factory):
    """(K, grid, P, part, warps that can rank, survivors) -> (block of every survivor in the row part, columns a block's tables hold)."""
    d = tmp_path_factory.mktemp("groups")
    src = d / "groups.cpp"
    src.write_text(r'''
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "celty_internal.h"
int main(int, char **v) {
    using namespace celty;
    const int K = atoi(v[1]), grid = atoi(v[2]), P = atoi(v[3]), s = atoi(v[4]), most = atoi(v[5]);
    const int warps = direct_rankers(direct_columns(K, grid / P), most == 16, most);          // (pairs of warps: all 16)
    std::vector<unsigned char> keep(K);
    if (fread(keep.data(), 1, K, stdin) != (size_t)K) return 1;
    const int nK = grid / P + (s < grid % P ? 1 : 0);
    const DirectGroups g = direct_groups(K, grid, P, warps, (K + grid / P - 1) / (grid / P) > 128);
    printf("%d %d\n", g.most, g.rankers);
    for (int b = 0; b < nK; ++b) {                       // as the kernel does it, block by block
        const DirectGroup q = direct_group(b, g.sizes[nK - grid / P]);
        for (int w = 0; w < g.rankers; ++w)
            for (int t = 32 * g.held * w, n = 0; t < 32 * g.held * (w + 1); ++t) {
                const int j = direct_held(t, q, nK, 1.f / (float)nK);
                if (j < 0) return 2;
                if (j < K && keep[j] && direct_taker(n++, w, 1.f / (float)g.rankers, q) == b - q.first) printf("%d %d\n", j, b);
            }
    }
}
''')
    exe = str(d / "groups")
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I",
                           os.path.join(ROOT, "paper_2608_01536_b200", "csrc"), "-o", exe, str(src)])

    def call(K, grid, P, part, warps, keep):
        out = subprocess.check_output([exe, str(K), str(grid), str(P), str(part), str(warps)], input=keep.astype(np.uint8).tobytes())
        rows = np.array(out.split(), dtype=np.int64).reshape(-1, 2)
        most, rankers = rows[0]
        assert 1 <= rankers <= warps - (2 if warps == 12 and K <= 46 * (grid // P) else 0)      # the others make the list
        taken = rows[1:]
        assert np.array_equal(np.sort(taken[:, 0]), np.flatnonzero(keep))      # every survivor once, and nothing else
        return taken[:, 1], most
    return call


@pytest.mark.parametrize("warps", [12, 16])
@pytest.mark.parametrize("grid,P", [(148, 1), (148, 2), (148, 3), (148, 5), (74, 1), (21, 2), (37, 4), (5, 5), (1, 1), (3, 2), (148, 147)])
def test_every_survivor_has_one_taker(takers, grid, P, warps):
    nK = grid // P
    rng = np.random.default_rng(grid * P)
    for K in sorted({1, 2, 3, nK, 2 * nK + 1, 31 * nK + 5, 56 * nK, 128 * nK - 1, 128 * nK, 128 * nK + 1, 171 * nK, 256 * nK + 3, 387 * nK, 512 * nK}):
        for part in {0, P - 1}:
            for keep in (np.ones(K, bool), rng.random(K) < 0.5, rng.random(K) < 0.03, np.zeros(K, bool)):
                own, most = takers(K, grid, P, part, warps, keep)
                counts = np.bincount(own, minlength=nK)
                assert counts.max(initial=0) <= most, (K, part, counts.max(), most)


# K and blocks per row part of 4096 x 4096, 5120 x 5120, 11008 x 4096, 2048 x 5504, 4096 x 11008, 8192 x 8192
@pytest.mark.parametrize("K,nK", [(4096, 74), (5120, 74), (4096, 49), (5504, 148), (11008, 148), (8192, 74), (13824, 148), (9700, 49), (28672, 74), (4096, 18)])
def test_groups_even_out_independent_survivors(takers, K, nK):
    """Survivors that fall independently, a share d of the columns: a group of s blocks has n d +- sqrt(n d (1 - d)) of its n
    columns, so a block of it has 1 / s of that, and one more per ranking warp at most where the warps' remainders meet; the
    warps' first blocks lie evenly, so two to three of these meet."""
    rng = np.random.default_rng(K + nK)
    for d in (0.1, 0.3, 0.5, 0.7):
        for _ in range(3):
            keep = rng.random(K) < d
            own, _ = takers(K, nK, 1, 0, 16, keep)
            counts = np.bincount(own, minlength=nK)
            columns = K / nK
            size = min(nK, max(3, int(512 // np.ceil(columns + 1))))            # three blocks share at least
            spread = np.sqrt(columns * d * (1 - d) / size)
            assert counts.max() <= keep.sum() / nK + 3.5 * spread + 3, (d, counts.max(), keep.sum() / nK, spread)
