"""GPU parity for small batches (N = 1 .. 8 activation vectors against one matrix) and for a layer sharded by
columns: the oracle is N independent plain products, and the plain product of the whole layer."""
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


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("variant", [0, 1])          # launches of the fused kernel / the widened kernels
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 8])
@pytest.mark.parametrize("M,K,d_w,d_a", [(1000, 520, 0.5, 0.5), (4096, 1024, 0.3, 0.2), (11008, 300, 0.5, 0.9),
                                         (28672, 96, 0.5, 0.5)])
def test_batch_matches_independent_products(N, M, K, d_w, d_a, variant):
    W = synth.weights(M + K, M, K)
    mask = synth.mask_bernoulli(M + K, M, K, d_w)
    X = np.stack([synth.activations(100 * n + K, K, "laplace") for n in range(N)])
    tau = synth.threshold_for_density(X[0], d_a)
    m = celty.Matrix(W, mask, device="cuda")
    m.set_launch(variant=variant)
    Y = m.spmspv_batch(_dev(X), tau, y=torch.full((N, M), 4.0, device="cuda"))
    torch.cuda.synchronize()
    got = Y.cpu().numpy().astype(np.float64)
    for n in range(N):
        y_ref, a_ref = orc.masked_gemv(W, mask, X[n], tau, threads=8)
        err = np.abs(got[n] - y_ref)
        assert np.all(err <= 2e-3 * a_ref + 1e-6), (n, float(err.max()))


def test_batch_integer_data_is_bit_exact_and_strided():
    """Small integers make every FP32 sum exact in any order; the batch rows sit in wider buffers (ldx > K, ldy > M);
    one vector has no survivor at all and one keeps everything."""
    M, K, N = 3000, 257, 6
    W = synth.integer_weights(9, M, K)
    mask = synth.mask_bernoulli(9, M, K, 0.6)
    X = np.stack([synth.integer_activations(20 + n, K) for n in range(N)])
    X[2] = 0
    X[4][X[4] == 0] = 1
    tau = 1.0
    xb = torch.zeros(N, K + 7 + 8 - (K + 7) % 8, dtype=torch.float16, device="cuda")
    xb[:, :K] = _dev(X)
    yb = torch.full((N, M + 5), -1.0, device="cuda")
    m = celty.Matrix(W, mask, device="cuda")
    m.spmspv_batch(xb[:, :K], tau, y=yb[:, :M])
    torch.cuda.synchronize()
    for n in range(N):
        y_ref, _ = orc.masked_gemv(W, mask, X[n], tau, threads=4)
        assert np.array_equal(yb[n, :M].cpu().numpy().astype(np.float64), y_ref), n
    assert torch.all(yb[:, M:] == -1.0)                           # nothing written past a row
    assert torch.count_nonzero(yb[2, :M]).item() == 0


@pytest.mark.parametrize("M,K,tile_rows", [(4096, 700, 0), (20000, 90, 0), (28672, 64, 0), (40, 33, 8), (9000, 257, 40)])
def test_batches_of_changing_size_on_one_handle(M, K, tile_rows):
    """Vectors that share a launch, on a handle that serves batches of every size and single vectors in turn (the
    tickets of one launch shape must not disturb another's), row parts that do not divide the blocks of a vector,
    more blocks than columns; integer data, so every sum is exact.  The list reported is the last vector's."""
    W = synth.integer_weights(5, M, K)
    mask = synth.mask_bernoulli(5, M, K, 0.5)
    X = np.stack([synth.integer_activations(40 + n, K) for n in range(8)])
    ref = np.stack([orc.masked_gemv(W, mask, X[n], 1.0, threads=8)[0] for n in range(8)])
    m = celty.Matrix(W, mask, tile_rows=tile_rows, device="cuda")
    wide = torch.zeros(8, (K + 7) // 8 * 8, dtype=torch.float16, device="cuda")
    wide[:, :K] = _dev(X)
    for N in (2, 8, 3, 1, 5, 8, 2, 7, 4, 6, 1, 3):
        y = torch.full((N, (M + 3) // 4 * 4), 9.0, device="cuda")[:, :M]
        m.spmspv_batch(wide[:N, :K], 1.0, y=y)
        torch.cuda.synchronize()
        assert m.last_status() == 0
        assert np.array_equal(y.cpu().numpy().astype(np.float64), ref[:N]), N
        idx, val = m.last_compaction()
        oi, ov, _ = orc.compact(X[N - 1], 1.0)
        assert np.array_equal(idx.cpu().numpy(), oi) and np.array_equal(val.cpu().numpy().view(np.uint16), ov), N
        y1 = m.spmspv(wide[N % 8, :K].contiguous(), 1.0)
        assert np.array_equal(y1.cpu().numpy().astype(np.float64), ref[N % 8]), N


@pytest.mark.parametrize("M,N,stuck", [(4096, 2, 1), (4096, 8, 0), (9000, 3, 2)])
def test_a_batch_wait_that_runs_out_is_reported_and_the_handle_recovers(M, N, stuck):
    """One vector's ticket is moved ahead by hand, so that some of its blocks wait for a count that never comes: the
    launch comes back by itself, last_status says CELTY_ETIMEOUT once and repairs the tickets, the other vectors of
    the launch are right, and so is the next batch."""
    K = 512
    W = synth.integer_weights(6, M, K)
    mask = synth.mask_bernoulli(6, M, K, 0.5)
    X = np.stack([synth.integer_activations(60 + n, K) for n in range(N)])
    ref = np.stack([orc.masked_gemv(W, mask, X[n], 1.0, threads=8)[0] for n in range(N)])
    m = celty.Matrix(W, mask, device="cuda")
    xd, y = _dev(X), torch.empty(N, M, device="cuda")
    m.spmspv_batch(xd, 1.0, y=y)
    torch.cuda.synchronize()
    assert m.last_status() == 0
    words = m._ws[:256].view(torch.int32)
    used = torch.nonzero(words[16:52]).flatten().tolist()        # tickets of batch launches stand at their block counts
    assert len(used) == N                                        # one launch served all of them
    grid = int(words[16 + used[stuck]].item())
    words[16 + used[stuck]] = grid + 5                           # five blocks will land in the other half
    m.set_wait_limit(2000)
    m.spmspv_batch(xd, 1.0, y=y)
    torch.cuda.synchronize()
    assert m.last_status() == -5 and m.last_status() == 0
    others = [n for n in range(N) if n != stuck]
    assert np.array_equal(y.cpu().numpy().astype(np.float64)[others], ref[others])
    m.set_wait_limit(0)
    for _ in range(2):
        m.spmspv_batch(xd, 1.0, y=y)
        assert m.last_status() == 0
        assert np.array_equal(y.cpu().numpy().astype(np.float64), ref)


def test_batch_argument_errors():
    m = celty.Matrix(synth.weights(1, 64, 40), None, device="cuda")
    x = torch.zeros(9, 40, dtype=torch.float16, device="cuda")
    with pytest.raises(celty.CeltyError):
        m.spmspv_batch(x, 0.1)                                    # more than 8 vectors
    col = celty.Matrix(synth.weights(1, 64, 40), None, layout=celty.LAYOUT_COLUMN, device="cuda")
    with pytest.raises(celty.CeltyError):
        col.spmspv_batch(x[:2], 0.1)


@pytest.mark.parametrize("world", [1, 2, 3, 5])
def test_column_shards_add_up_to_the_layer(world):
    """Every rank's share of a column-sharded layer, run one after the other on this GPU (no process group: the
    all-reduce is replaced by adding the partial results here), against the plain product of the whole layer."""
    M, K = 2049, 1003
    W = synth.weights(31, M, K)
    mask = synth.mask_bernoulli(31, M, K, 0.5)
    x = synth.activations(31, K, "laplace")
    tau = synth.threshold_for_density(x, 0.5)
    xd = _dev(x)
    total = torch.zeros(M, dtype=torch.float32, device="cuda")
    covered = []
    for rank in range(world):
        shard = celty.ColumnShard(W, mask, rank=rank, world=1 if world == 1 else world, device="cuda")
        covered.append((shard.k0, shard.k1))
        shard.world = 1                                           # no collective in this test
        total += shard.spmspv(xd, tau)
    assert covered[0][0] == 0 and covered[-1][1] == K
    assert all(a[1] == b[0] for a, b in zip(covered, covered[1:]))
    y_ref, a_ref = orc.masked_gemv(W, mask, x, tau, threads=8)
    assert np.all(np.abs(total.cpu().numpy().astype(np.float64) - y_ref) <= 2e-3 * a_ref + 1e-6)
