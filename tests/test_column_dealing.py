"""Which columns of x a block of k_spmspv_direct owns, evaluated by the library's own rule: every column has one owner and a
place among its 32-column chunks, and survivors that lie together in x are shared by the blocks.  No GPU needed."""
import os
import subprocess

import numpy as np
import pytest

from conftest import ROOT

CHUNKS = 4                                                # of 32 columns, at most


@pytest.fixture(scope="module")
def owners(tmp_path_factory):
    """(K, blocks) -> the block of every column, from a C++ program of a few lines around the library's direct_column."""
    d = tmp_path_factory.mktemp("dealing")
    src = d / "dealing.cpp"
    src.write_text('#include <cstdio>\n#include <cstdlib>\n#include "celty_internal.h"\n'
                   "int main(int, char **v) {\n"
                   "    const int K = atoi(v[1]), nK = atoi(v[2]), most = (K + nK - 1) / nK, places = (most + 31) / 32 * 32;\n"
                   "    for (int b = 0; b < nK; ++b)\n"
                   "        for (int i = 0; i < places; ++i) {\n"
                   "            const int j = celty::direct_column(i, b, nK, 1.f / (float)nK);\n"
                   '            if (j < K) printf("%d %d\\n", b, j);\n'
                   "        }\n}\n")
    exe = str(d / "dealing")
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I",
                           os.path.join(ROOT, "paper_2608_01536_b200", "csrc"), "-o", exe, str(src)])

    def call(K, nK):
        pairs = np.array(subprocess.check_output([exe, str(K), str(nK)], text=True).split(), dtype=np.int64).reshape(-1, 2)
        assert np.array_equal(np.sort(pairs[:, 1]), np.arange(K))        # every column once, and no other
        own = np.empty(K, np.int64)
        own[pairs[:, 1]] = pairs[:, 0]
        return own
    return call


@pytest.mark.parametrize("nK", [1, 2, 3, 18, 37, 49, 50, 74, 147, 148])
def test_every_column_has_one_owner(owners, nK):
    edges = {1, 2, 3, nK - 1, nK, nK + 1, 2 * nK + 1}
    for c in range(1, CHUNKS + 1):
        edges |= {32 * c * nK - 1, 32 * c * nK, 32 * (c - 1) * nK + 1}
    for K in sorted(e for e in edges if e >= 1):
        counts = np.bincount(owners(K, nK), minlength=nK)
        assert counts.max() - counts.min() <= 2, (K, counts.min(), counts.max())     # a run of two columns at most


def _structured(K, rng):
    """Activations of which a share survives, in patterns that layers see: some heads of an attention output zeroed, half of
    every head, a stretch of x, every second or 64th column."""
    i = np.arange(K)
    for width in (64, 128):
        heads = -(-K // width)
        for _ in range(4):
            alive = np.zeros(heads, bool)
            alive[rng.permutation(heads)[:heads // 2]] = True
            yield "heads", alive[i // width]
        yield "alternating heads", (i // width) % 2 == 0
        yield "half of every head", i % width < width // 2
    for part in (2, 4, 8):
        yield "a stretch", (i >= K // 2) & (i < K // 2 + K // part)
    for step in (2, 37, 64, 74, 148):
        yield "a comb", i % step == 1


# K and blocks per row part of 4096 x 4096, 5120 x 5120, 11008 x 4096, 2048 x 5504, 4096 x 11008, 8192 x 8192
@pytest.mark.parametrize("K,nK", [(4096, 74), (5120, 74), (4096, 49), (5504, 148), (11008, 148), (8192, 74)])
def test_structured_survivors_are_shared(owners, K, nK):
    """The busiest block sets a call's time.  If its runs of two columns survived or not independently of one another, half of
    them, the columns of a block would have the variance `mean`, and the busiest of 49 to 148 blocks 2.5 deviations more
    than the mean; structure may not cost more than that (and one run).  Runs of 32 columns gave it up to twice the mean."""
    own = owners(K, nK)
    for name, survives in _structured(K, np.random.default_rng(K)):
        counts = np.bincount(own[survives], minlength=nK)
        mean = survives.sum() / nK
        assert counts.max() <= mean + 2.5 * np.sqrt(mean) + 2, (name, mean, counts.max())
