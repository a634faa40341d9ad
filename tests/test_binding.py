"""What the binding passes to the library and what it refuses, without a GPU: calls go to a stand-in for the native module, or
to the module itself with a handle that has no device memory (the library then says CELTY_ESTATE before anything is launched)."""
from types import SimpleNamespace

import numpy as np
import pytest
import torch

from paper_2608_01536_b200 import build, celty, synth


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    celty.load()


def _matrix(M=64, K=48):
    return celty.Matrix(synth.integer_weights(3, M, K))


def test_batch_scratch_lies_beside_the_image(monkeypatch):
    """A call with an x of the wrong kind is refused, and what it leaves on the handle serves the next call."""
    seen = []

    def refuse(n, M, K, x, tau, y, stream, scratch):
        seen.append(scratch)
        raise AssertionError

    monkeypatch.setattr(celty, "_native", SimpleNamespace(spmspv_batch=refuse))
    m = _matrix()
    m._image = torch.empty(1, dtype=torch.uint8, device="meta")       # stands in for a GPU
    for _ in range(2):
        with pytest.raises(AssertionError):
            m.spmspv_batch(torch.zeros(2, m.K), 1.0)
    assert m._batch_scratch.device.type == "meta" and seen[0] is seen[1] is m._batch_scratch
    unbound = _matrix()
    with pytest.raises(AssertionError):
        unbound.spmspv_batch(torch.zeros(2, m.K), 1.0)
    assert unbound._batch_scratch is None
