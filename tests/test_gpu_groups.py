"""Products whose blocks share their columns' survivors in groups, at the edges of what a ranking lane holds (one, two or four
columns) and where the kernel that ranks all of x takes over (more than 512 columns per block, 384 where blocks left over can be shared)."""
import numpy as np
import pytest
import torch

from oracle import celty_oracle as orc
from paper_2608_01536_b200 import build, celty, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    assert torch.cuda.is_available(), "these tests need a CUDA device"
    celty.load()


# blocks of the launch; rows, rows per tile (row parts); columns per block of a row part: three members of a group need 512 / 3
# columns each (384 / 3 without warp pairs) for one column per lane, 341 (256) for two
@pytest.mark.parametrize("grid,M,tile_rows,columns", [(g, M, r, c) for g, M, r in ((5, 40, 0), (37, 300, 3), (148, 40, 0), (19, 1100, 4))
                                                       for c in (127, 128, 129, 170, 171, 256, 257, 341, 342, 512, 513)] +
                         [(148, 256, 1, c) for c in (127, 171, 257, 384, 385)])
def test_groups_at_their_edges(grid, M, tile_rows, columns):
    """Integer data, exact: three densities, survivors that lie together, none and all; the reported list; the call twice."""
    probe = celty.Matrix(synth.integer_weights(1, M, 8), None, tile_rows=tile_rows)
    parts = probe.row_map()[0]
    K = columns * (grid // parts)
    W = synth.integer_weights(columns + grid, M, K)
    mask = synth.mask_bernoulli(columns + grid, M, K, 0.4)
    m = celty.Matrix(W, mask, tile_rows=tile_rows, device="cuda")
    m.set_launch(grid=grid)
    plan, left = m.launch_plan(), grid % parts
    mixes = left > 0 and parts % left == 0 and parts // left * (grid // parts) <= 48       # left-over blocks can be shared
    assert plan["row_parts"] == parts and plan["kernel"] == ("k_spmspv_direct" if columns <= (384 if mixes else 512) else "k_spmspv_fused")
    rng = np.random.default_rng(columns)
    full = synth.integer_activations(9, K)
    full = np.where(full == 0, np.float16(1), full)               # 1 .. in magnitude
    for keep in (rng.random(K) < 0.5, rng.random(K) < 0.05, np.arange(K) < K // 3, np.zeros(K, bool), np.ones(K, bool)):
        x = np.where(keep, full, np.float16(0))
        ref, _ = orc.masked_gemv(W, mask, x, 0.5, threads=8)
        xd = torch.from_numpy(x).cuda()
        for _ in range(2):
            y = m.spmspv(xd, 0.5, y=torch.full((M,), 7.0, device="cuda"))
            assert np.array_equal(y.cpu().numpy().astype(np.float64), ref)
        oi, ov, _ = orc.compact(x, 0.5)
        gi, gv = m.last_compaction()
        assert np.array_equal(gi.cpu().numpy(), oi) and np.array_equal(gv.cpu().numpy().view(np.uint16), ov)
        if K <= 32768:
            assert np.array_equal(m.spmspv_static(xd, 0.5).cpu().numpy().astype(np.float64), ref)
    assert m.last_status() == 0


# a warp per column (28 of 32 in flight), several, one warp given up for the list; grids of fewer and more blocks than SMs; the last size
# that is dealt and the first that is not (129 columns per block, a column of more passes than there are others in flight)
@pytest.mark.parametrize("M,K,d_w,grid", [(3, 5, 1.0, 0), (100, 9000, 0.5, 0), (256, 150, 1.0, 0), (300, 148 * 128, 0.5, 0), (300, 148 * 128 + 1, 0.5, 0),
                                          (4096, 4096, 0.5, 0), (2048, 3001, 0.9, 0), (1000, 997, 0.3, 5), (2000, 800, 0.5, 400), (7000, 2300, 0.5, 0),
                                          (12000, 600, 0.5, 0), (20000, 500, 0.5, 0), (8100, 64, 1.0, 1), (40, 200, 0.02, 2)])
def test_whole_columns_dealt_to_groups(M, K, d_w, grid):
    """Integer data, exact: half, few, none and all of the activations, and survivors that lie together; the reported list."""
    W = synth.integer_weights(M + K, M, K)
    mask = synth.mask_bernoulli(M + K, M, K, d_w) if d_w < 1 else np.ones((M, K), np.uint8)
    m = celty.Matrix(W, mask, layout=celty.LAYOUT_COLUMN, device="cuda")
    m.set_launch(grid=grid)
    rng = np.random.default_rng(M + K)
    full = synth.integer_activations(10, K)
    full = np.where(full == 0, np.float16(-1), full)
    for keep in (rng.random(K) < 0.5, rng.random(K) < 0.05, np.arange(K) < K // 3, np.zeros(K, bool), np.ones(K, bool)):
        x = np.where(keep, full, np.float16(0))
        ref, _ = orc.masked_gemv(W, mask, x, 0.5, threads=8)
        oi, ov, _ = orc.compact(x, 0.5)
        xd = torch.from_numpy(x).cuda()
        for _ in range(2):
            y = m.spmspv(xd, 0.5, y=torch.full((M,), 7.0, device="cuda"))
            assert np.array_equal(y.cpu().numpy().astype(np.float64), ref)
            gi, gv = m.last_compaction()
            assert np.array_equal(gi.cpu().numpy(), oi) and np.array_equal(gv.cpu().numpy().view(np.uint16), ov.view(np.uint16))
    assert m.last_status() == 0
