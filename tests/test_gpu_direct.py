"""Products of layers whose thread blocks own few columns, dealt to them whatever x is, against the oracle and against the
kernel that ranks the survivors (variant 256): the edges of 32, 64, 96 and 128 columns per block, row parts of unequal block
counts, more blocks than columns, survivors that cluster in x."""
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


def _clusters(K, seed):
    """Integer activations whose survivors lie everywhere, in one eighth of x, in every 37th place, nowhere, everywhere and
    all kept."""
    x = synth.integer_activations(seed, K)
    eighth, comb, full = np.zeros_like(x), np.zeros_like(x), x.copy()
    eighth[K // 2:K // 2 + max(1, K // 8)] = 3
    comb[::37] = -2
    full[full == 0] = 1
    return [x, eighth, comb, np.zeros_like(x), full]


# tile rows of 2 make 4 row parts of 37 blocks, of 3 make 3 parts of 50, 49 and 49; without, one part of 148
@pytest.mark.parametrize("M,tile_rows,K", [(200, 2, k) for k in (1, 36, 37, 38, 1184, 1185, 2368, 2369, 3553, 4736, 4737)] +
                         [(257, 3, k) for k in (49, 50, 1568, 1569, 3137, 6272, 6273)] +
                         [(40, 0, k) for k in (147, 149, 4736, 4737, 9473, 18944, 18945)])
def test_columns_dealt_to_blocks(M, tile_rows, K):
    W = synth.integer_weights(M + K, M, K)
    mask = synth.mask_bernoulli(M + K, M, K, 0.4)
    m = celty.Matrix(W, mask, tile_rows=tile_rows, device="cuda")
    for x in _clusters(K, K):
        y_ref, _ = orc.masked_gemv(W, mask, x, 0.5, threads=8)
        oi, ov, _ = orc.compact(x, 0.5)
        xd = torch.from_numpy(x).cuda()
        order = np.random.default_rng(K).permutation(oi.size)         # a list may come in any order
        idx = torch.from_numpy(np.append(oi[order], 0).astype(np.int32)).cuda()
        val = torch.from_numpy(np.append(ov[order], 0).astype(np.uint16).view(np.int16)).cuda()
        n = torch.tensor([oi.size], dtype=torch.int32, device="cuda")
        for variant in (0, 256, 16, 32):
            m.set_launch(variant=variant)
            y = m.spmspv(xd, 0.5, y=torch.full((M,), 5.0, device="cuda"))
            gi, gv = m.last_compaction()
            assert np.array_equal(y.cpu().numpy().astype(np.float64), y_ref), variant
            assert np.array_equal(gi.cpu().numpy(), oi) and np.array_equal(gv.cpu().numpy().view(np.uint16), ov), variant
            y = m.spmspv_list(idx, val, n, y=torch.full((M,), 6.0, device="cuda"))
            assert np.array_equal(y.cpu().numpy().astype(np.float64), y_ref), variant
            assert m.last_status() == 0
        y = m.spmspv_static(xd, 0.5, y=torch.full((M,), 7.0, device="cuda"))
        assert np.array_equal(y.cpu().numpy().astype(np.float64), y_ref)
