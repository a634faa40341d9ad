"""The kernel that ranks the survivors, on layers where it is the default (more than 512 columns per thread block, 384 where left-over
blocks can be shared) and in the builds that the launch choices ask for, and both kernels where what they decide is their own
code: thresholds, batches, waits that run out."""
import numpy as np
import pytest
import torch

from conftest import lane_tile_rows
from oracle import celty_oracle as orc
from paper_2608_01536_b200 import build, celty, synth

pytestmark = pytest.mark.gpu

RANKED, DIRECT = "k_spmspv_fused", "k_spmspv_direct"


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    assert torch.cuda.is_available(), "these tests need a CUDA device"
    celty.load()


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _layer(seed, M, K, **kw):
    W = synth.integer_weights(seed, M, K)
    mask = synth.mask_bernoulli(seed, M, K, 0.5)
    return W, mask, celty.Matrix(W, mask, device="cuda", **kw)


SPECIAL_X = np.array([0x0000, 0x8000, 0x7E00, 0xFE00, 0x7C00, 0xFC00, 0x0001, 0x8001, 0x03FF, 0x83FF, 0x0400, 0x8400,
                      0x7BFF, 0xFBFF, 0x3C00, 0xBC00, 0x3C01, 0x3BFF, 0x3800, 0xB800], np.uint16)


@pytest.mark.parametrize("tiles,empty,kernel", [(32, 3, DIRECT), (256, 3, DIRECT), (992, 3, DIRECT), (32, 20001, DIRECT),
                                                (992, 1300, RANKED), (32, 76001, RANKED)])
def test_special_values_reach_y_through_every_kernel(tiles, empty, kernel):
    """Every column of W fills one tile of 8 rows with ones, so y shows which columns the product took: +-0, NaNs, infinities,
    subnormals and the neighbours of 1 against thresholds that are 0, below the smallest subnormal, on FP16 values, between
    two of them, the largest finite value and beyond.  (Full groups of 8 entries: the zeros that fill up a group would be
    NaN beside an infinity.)  Empty columns at the end make the last keep word a short one."""
    M, K = 8 * tiles, tiles + empty
    rows = lane_tile_rows(M, M // 256, 8, 8)                      # tile, local row -> row
    W = np.zeros((M, K), np.float16)
    W[rows, np.arange(tiles)[:, None]] = 1
    x = synth.activations(K + 3, K, "laplace").view(np.uint16).copy()
    x[(np.arange(SPECIAL_X.size) * 37) % tiles] = SPECIAL_X
    x[-3:] = SPECIAL_X[2:5]                                       # of empty columns as well
    x = x.view(np.float16)
    m = celty.Matrix(W, None, tile_rows=8, device="cuda")
    assert m.row_map() == (M // 256, 8, 8) and m.info().n_pad == 0
    xd = _dev(x)
    wide = torch.zeros(2, (K + 7) // 8 * 8, dtype=torch.float16, device="cuda")
    wide[:, :K] = xd
    yb = torch.empty(2, M, device="cuda")
    for variant in (0, 128, 256, 16, 32, 2):
        m.set_launch(variant=variant)
        assert m.launch_plan()["kernel"] == (kernel if variant in (0, 16, 32) else RANKED)
        for tau in (0.0, 1e-8, 5.9604645e-08, 0.99975586, 1.0, 1.0004883, 0.7, 65504.0, 65519.9, 1e5):
            with np.errstate(invalid="ignore"):
                keep = ~(np.abs(x.astype(np.float32)) <= np.float32(tau))
            want = np.empty(M, np.float32)
            want[rows] = np.where(keep, x.astype(np.float32), np.float32(0))[:tiles, None]
            ys = [m.spmspv(xd, tau, y=torch.full((M,), 3.0, device="cuda"))]
            oi, ov, _ = orc.compact(x, tau)
            gi, gv = m.last_compaction()
            assert np.array_equal(gi.cpu().numpy(), oi) and np.array_equal(gv.cpu().numpy().view(np.uint16), ov), (variant, tau)
            if variant != 2:                                      # lists: with the bulk reduce-add merge only
                n = torch.tensor([oi.size], dtype=torch.int32, device="cuda")
                ys.append(m.spmspv_list(_dev(np.append(oi, 0).astype(np.int32)), _dev(np.append(ov, 0).astype(np.uint16).view(np.int16)), n))
            if variant == 0:
                ys += ([m.spmspv_static(xd, tau)] if K <= 32768 else []) + list(m.spmspv_batch(wide[:, :K], tau, y=yb))
            for k, y in enumerate(ys):
                assert np.array_equal(y.cpu().numpy(), want, equal_nan=True), (variant, tau, k)
        assert m.last_status() == 0


# blocks of a vector at the edges of 32, 64, 96, 128 and 512 columns per block, or of 20 000 / rows per lane, beyond which survivors are ranked
@pytest.mark.parametrize("N,M,tile_rows,K", [(2, 40, 0, 74 * 32 * c + e) for c in (1, 2, 3, 4) for e in (0, 1)] +
                         [(5, 40, 0, 29 * 128 + e) for e in (-1, 1)] + [(3, 200, 2, 12 * 128 + e) for e in (0, 1)] +
                         [(2, 40, 0, 74 * 512 + e) for e in (0, 1)] + [(8, 4096, 128, 18 * 156 + e) for e in (0, 1)] +
                         [(4, 4096, 0, 4096), (3, 4096, 0, 4096), (8, 2048, 0, 4096), (8, 300, 0, 40000), (4, 9000, 0, 3000)])
def test_batches_on_both_sides_of_the_line(N, M, tile_rows, K):
    """Integer data, exact; also with two teams per block, so that a team has more columns than it looks up at once."""
    W, mask, m = _layer(M + N, M, K, tile_rows=tile_rows)
    X = np.stack([synth.integer_activations(90 + n, K) for n in range(N)])
    X[0, :K // 2] = 0                                             # survivors to one side
    ref = np.stack([orc.masked_gemv(W, mask, X[n], 1.0, threads=8)[0] for n in range(N)])
    wide = torch.zeros(N, (K + 7) // 8 * 8, dtype=torch.float16, device="cuda")
    wide[:, :K] = _dev(X)
    oi, ov, _ = orc.compact(X[N - 1], 1.0)
    for variant, groups in ((0, 0), (128, 0), (0, 2), (16, 2), (32, 1)):
        m.set_launch(variant=variant, groups=groups)
        plan = m.launch_plan()
        columns = -(-K // (148 // N // plan["row_parts"]))
        most = max(128, min(512, 20000 // m.row_map()[1]))
        assert plan["batch_kernels"][N] == (DIRECT if columns <= most and variant != 128 else RANKED)
        y = torch.full((N, (M + 3) // 4 * 4), 9.0, device="cuda")[:, :M]
        for _ in range(2):
            m.spmspv_batch(wide[:, :K], 1.0, y=y)
        assert np.array_equal(y.cpu().numpy().astype(np.float64), ref), variant
        idx, val = m.last_compaction()
        assert np.array_equal(idx.cpu().numpy(), oi) and np.array_equal(val.cpu().numpy().view(np.uint16), ov), variant
        assert m.last_status() == 0


# (tile_rows 64: two row parts; 2: five; 1: eight, between which four blocks left over are shared)
@pytest.mark.parametrize("M,K,tile_rows,grid,variant,kernel", [
    (300, 20000, 0, 0, 0, DIRECT), (4096, 12000, 64, 0, 16, DIRECT), (4096, 12000, 64, 0, 32, DIRECT), (300, 15000, 2, 0, 0, RANKED),
    (300, 15000, 2, 0, 16, RANKED), (300, 15000, 2, 0, 32, RANKED), (4096, 5200, 64, 20, 16, RANKED), (4096, 5200, 64, 20, 32, RANKED),
    (256, 7000, 1, 0, 0, RANKED)])
def test_a_wait_that_runs_out_is_reported_and_the_handle_recovers(M, K, tile_rows, grid, variant, kernel):
    """The ticket that tells a block when the others have cleared their shares of y is moved ahead by hand, so that five
    blocks wait for a count that never comes: the launch comes back, the status says so once, the next call is right."""
    W, mask, m = _layer(61, M, K, tile_rows=tile_rows)
    m.set_launch(variant=variant, grid=grid)
    plan = m.launch_plan()
    assert plan["kernel"] == kernel and plan["parts_per_spare_block"] == (2 if tile_rows == 1 else 1)
    x = synth.integer_activations(62, K)
    y_ref, _ = orc.masked_gemv(W, mask, x, 1.0, threads=8)
    xd = _dev(x)
    y = m.spmspv(xd, 1.0)
    torch.cuda.synchronize()
    tickets, grid = m._ws[8:16].view(torch.int32), plan["grid"]
    assert int(tickets[0].item()) == grid
    tickets[0] = grid + 5
    m.set_wait_limit(2000)
    m.spmspv(xd, 1.0, y=y)
    torch.cuda.synchronize()
    assert m.last_status() == -5 and m.last_status() == 0
    m.set_wait_limit(0)
    for _ in range(2):
        assert np.array_equal(m.spmspv(xd, 1.0).cpu().numpy().astype(np.float64), y_ref)
        assert m.last_status() == 0


@pytest.mark.parametrize("M,K,tile_rows,grid,variant,depth,kernel", [
    (300, 20000, 0, 0, 0, 0, DIRECT), (4096, 12000, 64, 0, 16, 0, DIRECT), (4096, 12000, 64, 0, 16, 4, DIRECT), (4096, 12000, 64, 0, 32, 0, DIRECT),
    (300, 15000, 2, 0, 0, 0, RANKED), (300, 15000, 2, 0, 16, 0, RANKED), (300, 15000, 2, 0, 32, 0, RANKED), (4096, 5200, 64, 20, 16, 0, RANKED),
    (4096, 5200, 64, 20, 16, 4, RANKED), (4096, 5200, 64, 20, 32, 0, RANKED), (256, 7000, 1, 0, 0, 0, RANKED)])
def test_the_shortest_wait_limit(M, K, tile_rows, grid, variant, depth, kernel):
    """One poll per wait in single, list, batch and static calls of layers with many columns per block: the kernels come back,
    what they asked for has landed before their blocks end, and the handle is right again after last_status.  In the call
    without a status word every row is right or NaN."""
    W, mask, m = _layer(63, M, K, tile_rows=tile_rows)
    beside = m.clone("cuda")
    m.set_launch(variant=variant, depth=depth, grid=grid)
    plan = m.launch_plan()
    assert plan["kernel"] == kernel and plan["batch_kernels"][4] == RANKED
    x = synth.integer_activations(64, K)
    y_ref, _ = orc.masked_gemv(W, mask, x, 1.0, threads=8)
    oi, ov, _ = orc.compact(x, 1.0)
    xd, idx, val, n = _dev(x), _dev(oi), _dev(ov.view(np.int16)), _dev(np.array([oi.size], np.int32))
    xb, yb = xd.repeat(4, 1).contiguous(), torch.empty(4, M, device="cuda")
    cold = torch.empty(1 << 26, dtype=torch.float32, device="cuda")
    for _ in range(3):
        cold.zero_()                                              # the first copies come from memory, not from L2
        m.set_wait_limit(1)
        m.spmspv(xd, 1.0)
        m.spmspv_list(idx, val, n)
        m.spmspv_batch(xb, 1.0, y=yb)
        y = beside.spmspv(xd, 1.0)
        assert m.last_status() in (0, -5)
        assert beside.last_status() == 0 and np.array_equal(y.cpu().numpy().astype(np.float64), y_ref)
        cold.zero_()
        ys = m.spmspv_static(xd, 1.0).cpu().numpy().astype(np.float64)
        assert np.all(np.isnan(ys) | (ys == y_ref))
        m.set_wait_limit(0)
        for got in (m.spmspv(xd, 1.0), m.spmspv_static(xd, 1.0), *m.spmspv_batch(xb, 1.0, y=yb)):
            assert np.array_equal(got.cpu().numpy().astype(np.float64), y_ref)
        assert m.last_status() == 0
