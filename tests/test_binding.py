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


def test_vectors_in_pageable_host_memory_are_refused():
    """A kernel does not reach them.  (The handle has no device memory: what is let through ends with the library's status.)"""
    from paper_2608_01536_b200 import _celty_torch as calls
    M, K = 64, 48
    n, stream = _matrix(M, K)._n, SimpleNamespace(cuda_stream=0)
    x, y, f = torch.zeros(K, dtype=torch.float16), torch.zeros(M), torch.zeros(M, dtype=torch.float16)
    gate_up, idx, val, count = torch.zeros(2 * K), torch.zeros(K, dtype=torch.int32), x, torch.zeros(1, dtype=torch.int32)
    scratch = torch.zeros(1 << 16, dtype=torch.uint8)
    for out in (y, None):
        for call, args in ((calls.spmspv, (n, M, K, x, 1.0, out, stream)),
                           (calls.spmspv_static, (n, M, K, x, 1.0, out, stream, scratch)),
                           (calls.spmspv_ex, (n, M, K, x, 1.0, out, stream, f, None)),
                           (calls.spmspv_swiglu, (n, M, K, gate_up, 1.0, out, stream, x, f)),
                           (calls.spmspv_list, (n, M, idx, val, count, out, stream, None)),
                           (calls.spmspv_batch, (n, M, K, x[None], 1.0, None if out is None else out[None], stream, scratch))):
            with pytest.raises(AssertionError):
                call(*args)


def test_a_matrix_that_was_given_back_has_no_handle():
    """Calls on it reach the library with null, which it refuses, and not with memory that is no longer the matrix's."""
    m = _matrix()
    assert m._n == m._h.value
    m.__del__()
    assert m._h is None and m._n is None


def test_the_module_is_tied_to_its_torch(monkeypatch):
    """With another torch than the one it was built against it is built again, and is not called."""
    assert not build.needs_build()
    monkeypatch.setattr(torch, "__version__", torch.__version__ + ".other")
    assert build.needs_build()
    monkeypatch.setattr(celty, "_native", None)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: None)
    with pytest.raises(RuntimeError, match="built with torch"):
        celty._calls()
