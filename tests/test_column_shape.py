"""How the COLUMN product splits its work (warps per column, columns in flight, look-up batches, where the list comes
from), evaluated by the library's own rule for B200: the cases of the GPU test reach the edges they are there for, and
every height the library takes has a shape.  No GPU needed."""
import os
import subprocess

import numpy as np
import pytest

from conftest import ROOT
from paper_2608_01536_b200 import build, celty, synth

SMS, SMEM = 148, 232448                 # B200: SMs, bytes of shared memory a block can ask for

# M, K, d_w, d_a, grid (0: one block per SM) -> warps per column, columns in flight, columns looked up at a time, list by
# the blocks themselves
COLUMN_EDGES = [
    ((256, 150, 1.0, 1.0, 0), (2, 2, 3, 1)),             # every column exactly one chunk of 256 entries
    ((257, 40, 1.0, 1.0, 0), (2, 1, 2, 1)),              # ... and one entry more
    ((100, 9000, 0.5, 0.5, 0), (1, 32, 62, 1)),          # one warp per column, 32 of them in flight
    ((480, 90, 1.0, 1.0, 3), (2, 15, 31, 1)),            # fifteen groups (the named barriers there are), three blocks
    ((511, 2000, 0.9, 0.9, 3), (1, 32, 668, 1)),         # hundreds of columns to a block, two passes over each
    ((3, 5000, 0.5, 0.5, 1), (1, 32, 1024, 1)),          # one block, tiny columns, several batches of look-ups
    ((8100, 64, 1.0, 1.0, 0), (32, 1, 2, 1)),            # 32 warps on one column, one pass
    ((8192, 64, 1.0, 1.0, 0), (17, 1, 2, 1)),            # two passes over a column, the second not full
    ((8200, 64, 1.0, 1.0, 0), (17, 1, 2, 1)),            # ... one group of entries more
    ((8448, 64, 1.0, 1.0, 0), (17, 1, 2, 1)),            # ... a whole chunk more
    ((49152, 37, 0.4, 1.0, 0), (26, 1, 2, 1)),           # the tallest accumulator
    ((40001, 300, 0.02, 0.7, 0), (12, 1, 4, 1)),         # padding entries; M not a multiple of 4
    ((2, 262145, 0.5, 0.001, 0), (1, 32, 1024, 0)),      # the list comes from the compaction kernel
    ((2, 262145, 0.5, 0.02, 1), (1, 32, 1024, 0)),       # ... and is looked up in several batches
    ((60, 262144, 0.05, 0.01, 1), (1, 32, 1024, 1)),    # the longest x thresholded by the blocks
]


@pytest.fixture(scope="module")
def shape(tmp_path_factory):
    """column_shape of the library, called from a C++ program of a few lines."""
    build.build()
    d = tmp_path_factory.mktemp("shape")
    src = d / "shape.cpp"
    src.write_text('#include <cstdio>\n#include <cstdlib>\n#include "celty_internal.h"\n'
                   "int main(int n, char **v) {\n"
                   "    for (int i = 1; i + 2 < n; i += 4) {\n"
                   "        const auto s = celty::column_shape(atoll(v[i]), atoll(v[i + 1]), (size_t)atoll(v[i + 2]), %d, atoi(v[i + 3]));\n"
                   '        printf("%%d %%d %%d %%d %%zu\\n", s.W, s.groups, s.cap, s.own_list, s.smem);\n'
                   "    }\n}\n" % SMEM)
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I",
                           os.path.join(ROOT, "paper_2608_01536_b200", "csrc"), "-o", str(d / "shape"), str(src)])

    def call(*queries):                                   # (M, K, bytes of the entry stream, grid) each
        out = subprocess.check_output([str(d / "shape")] + [str(int(a)) for q in queries for a in q], text=True)
        return [tuple(int(a) for a in line.split()) for line in out.splitlines()]
    return call


@pytest.mark.parametrize("case,want", COLUMN_EDGES)
def test_the_gpu_cases_reach_the_edges_they_name(shape, case, want):
    M, K, d_w, _, grid = case
    W = synth.integer_weights(21, M, K)
    mask = synth.mask_bernoulli(21, M, K, d_w) if d_w < 1 else np.ones((M, K), np.uint8)
    image, stream_offset = celty.Matrix(W, mask, layout=celty.LAYOUT_COLUMN).host_image()
    (got,) = shape((M, K, image.size - stream_offset, grid or SMS))
    assert got[:4] == want
    assert got[4] <= SMEM


def test_every_height_has_a_shape(shape):
    """Up to the most rows a handle can have, for short and very long x, sparse and dense columns, any grid."""
    queries = [(M, K, round(d * M / 8 + 1) * 20 * K, grid) for M in (1, 1000, 30000, 45000, 49149, 49152)
               for K in (1, 500, 200_000, 262_144, 262_145, 2_000_000) for d in (0.01, 1.0) for grid in (1, SMS, 400)]
    for q, s in zip(queries, shape(*queries)):
        W, groups, cap, _, smem = s
        assert 1 <= W <= 32 and groups >= 1 and W * groups <= 32 and (W == 1 or groups <= 15) and cap >= 1, (q, s)
        assert smem <= SMEM, (q, s)
