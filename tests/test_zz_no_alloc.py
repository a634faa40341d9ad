"""celty_spmspv_static: the entry point for callers that cannot allocate device memory (a stream capture
in progress, a pool that owns the whole device, a host application that forbids allocations on its
inference path).  Its scratch is a fixed array inside the library, so the call takes only the packed image,
x and y.  This file is collected last on purpose: the array is shared by every call in the process.

The check: two calls in a row must each reproduce what the existing entry point (celty_spmspv, with its
caller-provided workspace) returns, within the bound the parity tests use.
"""
import ctypes

import numpy as np
import pytest
import torch

from conftest import hold_some_sms
from oracle import celty_oracle as orc
from paper_2608_01536_b200 import build, celty, synth

pytestmark = pytest.mark.gpu


def test_static_scratch_entry_point_matches_the_workspace_entry_point_twice():
    build.build()
    assert torch.cuda.is_available(), "needs a CUDA device"
    M, K = 4096, 1536
    W = synth.weights(77, M, K)
    mask = synth.mask_bernoulli(77, M, K, 0.5)
    m = celty.Matrix(W, mask, device="cuda")
    # bound of the parity tests: 2e-3 * sum_j |W_ij x_j| + 1e-6 per element
    for call, seed in enumerate((1, 2)):                      # second call: other survivors, same scratch
        x = synth.activations(seed, K, "laplace")
        tau = synth.threshold_for_density(x, 0.5 if call == 0 else 0.3)
        xd = torch.from_numpy(x).cuda()
        y_ws = m.spmspv(xd, tau)                              # existing entry point
        y_st = m.spmspv_static(xd, tau, y=torch.full((M,), 3.0, device="cuda"))
        torch.cuda.synchronize()
        y_ref, a_ref = orc.masked_gemv(W, mask, x, tau, threads=8)
        bound = 2e-3 * a_ref + 1e-6
        got = y_st.cpu().numpy().astype(np.float64)
        # against the existing entry point ...
        assert np.all(np.abs(got - y_ws.cpu().numpy().astype(np.float64)) <= bound), call
        # ... and against the definition itself
        assert np.all(np.abs(got - y_ref) <= bound), call
        assert torch.count_nonzero(y_st).item() > 0


def test_static_scratch_entry_point_leaves_device_memory_alone():
    """The point of the entry point: a call takes no device memory.  The free-memory figure of the
    driver must be the same before and after a call (the first call on the device has already looked
    up the array's address; outputs are allocated beforehand)."""
    build.build()
    M, K = 2048, 1024
    W = synth.weights(78, M, K)
    mask = synth.mask_bernoulli(78, M, K, 0.5)
    m = celty.Matrix(W, mask, device="cuda")
    x = synth.activations(3, K, "laplace")
    tau = synth.threshold_for_density(x, 0.5)
    xd = torch.from_numpy(x).cuda()
    y = torch.empty(M, dtype=torch.float32, device="cuda")
    m.spmspv_static(xd, tau, y=y)                             # set-up call
    torch.cuda.synchronize()
    free_before = torch.cuda.mem_get_info()[0]
    m.spmspv_static(xd, tau, y=y)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free_before
    y_ref, a_ref = orc.masked_gemv(W, mask, x, tau, threads=8)
    assert np.all(np.abs(y.cpu().numpy().astype(np.float64) - y_ref) <= 2e-3 * a_ref + 1e-6)


def test_static_and_two_launch_entry_points_share_one_kernel_attribute():
    """Entry points that launch one kernel with different amounts of dynamic shared memory: the lane-tile kernel of two
    launches, which the third handle's static call falls back to as well, and the fused kernel of the other static
    calls and of a handle without variant 1.  Interleaving them must not leave any with a stale idea of what the
    runtime currently allows."""
    build.build()
    K = 256
    mats = []
    for M, kw in ((4096, {}), (12288, {}), (40000, dict(tile_rows=240, slabs_per_block=6)), (1000, {})):
        W = synth.weights(80 + M, M, K)
        mask = synth.mask_bernoulli(80 + M, M, K, 0.5)
        m = celty.Matrix(W, mask, device="cuda", **kw)
        m.set_launch(variant=0 if M == 1000 else 1)
        mats.append((m, W, mask))
    with pytest.raises(celty.CeltyError):
        mats[2][0].launch_plan()                              # no room for the fused kernel: the static call's other route
    x = synth.activations(5, K, "laplace")
    tau = synth.threshold_for_density(x, 0.5)
    xd = torch.from_numpy(x).cuda()
    small, big, tall, fused = 0, 1, 2, 3
    for which, static in ((small, False), (tall, True), (big, False), (fused, False), (big, True), (small, False),
                          (small, True), (tall, False), (fused, True), (big, False), (tall, True), (fused, False)):
        m, W, mask = mats[which]
        y = m.spmspv_static(xd, tau) if static else m.spmspv(xd, tau)
        torch.cuda.synchronize()
        y_ref, a_ref = orc.masked_gemv(W, mask, x, tau, threads=8)
        assert np.all(np.abs(y.cpu().numpy().astype(np.float64) - y_ref) <= 2e-3 * a_ref + 1e-6), (W.shape, static)


@pytest.mark.parametrize("M,K,kw", [(1, 1, {}), (33, 8, {}), (1025, 2049, {}), (49152, 16, {}), (300, 32768, {}),
                                     (28672, 64, {}), (20000, 100, {}), (3000, 40, dict(tile_rows=240)),
                                     (7000, 40, dict(tile_rows=200, slabs_per_block=2)),
                                     (40000, 24, dict(tile_rows=240, slabs_per_block=6))])   # the last: two launches
def test_static_entry_point_over_its_range(M, K, kw):
    """Integer data, so every sum is exact: the smallest sizes, the limits, row parts that leave blocks over, and a
    shape that the single-launch kernel has no room for; the handle's launch choices change nothing."""
    build.build()
    W = synth.integer_weights(3, M, K)
    mask = synth.mask_bernoulli(3, M, K, 0.6)
    x = synth.integer_activations(4, K)
    m = celty.Matrix(W, mask, device="cuda", **kw)
    y_ref, _ = orc.masked_gemv(W, mask, x, 1.0, threads=8)
    xd = torch.from_numpy(x).cuda()
    for variant in (0, 2, 1, 0):
        m.set_launch(variant=variant)
        y = m.spmspv_static(xd, 1.0, y=torch.full((M,), 7.0, device="cuda"))
        assert np.array_equal(y.cpu().numpy().astype(np.float64), y_ref), variant


def test_static_scratch_entry_point_rejects_what_it_cannot_hold():
    build.build()
    lib = celty.load()
    wide = celty.Matrix(np.ones((4, 32769), np.float16))       # K beyond the fixed array
    p16 = ctypes.c_void_p(16)
    assert lib.celty_spmspv_static(wide._h, p16, p16, 0.0, p16, None) == -7
    assert lib.celty_strerror(-7) == b"size exceeds the fixed scratch of the no-allocation entry point"
    col = celty.Matrix(np.ones((4, 4), np.float16), layout=celty.LAYOUT_COLUMN)
    assert lib.celty_spmspv_static(col._h, p16, p16, 0.0, p16, None) == -1
    ok = celty.Matrix(np.ones((4, 4), np.float16))
    assert lib.celty_spmspv_static(ok._h, p16, p16, -1.0, p16, None) == -1
    assert lib.celty_spmspv_static(ok._h, None, p16, 0.0, p16, None) == -1


def test_static_entry_point_behind_the_kernel_that_writes_the_image():
    """The image need not come from a copy: here the kernel right before the call in the stream writes it."""
    build.build()
    M, K = 4096, 4096
    W = synth.integer_weights(6, M, K)
    mask = synth.mask_bernoulli(6, M, K, 0.5)
    x = synth.integer_activations(7, K)
    m = celty.Matrix(W, mask, device="cuda")
    y_ref, _ = orc.masked_gemv(W, mask, x, 1.0, threads=8)
    xd = torch.from_numpy(x).cuda()
    scrambled = m._image ^ 0x5A
    key = torch.full_like(scrambled, 0x5A)
    for _ in range(5):
        m._image.zero_()
        torch.bitwise_xor(scrambled, key, out=m._image)
        y = m.spmspv_static(xd, 1.0)
        assert np.array_equal(y.cpu().numpy().astype(np.float64), y_ref)


def test_static_call_needs_only_the_sms_that_are_free():
    """No block of the call waits for another: while a kernel of another stream keeps 39 SMs, the call's blocks run on
    the others, one after another where they have to, and the call is over before that kernel is."""
    build.build()
    M, K = 4096, 2048
    W = synth.integer_weights(8, M, K)
    mask = synth.mask_bernoulli(8, M, K, 0.5)
    x = synth.integer_activations(9, K)
    m = celty.Matrix(W, mask, device="cuda")
    y_ref, _ = orc.masked_gemv(W, mask, x, 1.0, threads=8)
    xd = torch.from_numpy(x).cuda()
    y = torch.full((M,), 7.0, device="cuda")
    m.spmspv_static(xd, 1.0, y=torch.empty_like(y))            # everything loaded
    torch.cuda.synchronize()
    other, mine = torch.cuda.Stream(), torch.cuda.Stream()
    holder, held = hold_some_sms(celty, synth, other)
    m.spmspv_static(xd, 1.0, y=y, stream=mine)
    mine.synchronize()
    assert not held.query()
    held.synchronize()
    assert holder.last_status() == -5
    assert np.array_equal(y.cpu().numpy().astype(np.float64), y_ref)


@pytest.mark.parametrize("layout", [celty.LAYOUT_LANE_TILE, celty.LAYOUT_COLUMN])
def test_calls_behind_a_clearing_kernel_in_a_captured_graph(layout):
    """The calls that clear y by a kernel of their own, captured after one call each and replayed with other activations
    in the same place; other y contents before every replay."""
    build.build()
    M, K = 3000, 1111
    W = synth.integer_weights(12, M, K)
    mask = synth.mask_bernoulli(12, M, K, 0.5)
    m = celty.Matrix(W, mask, layout=layout, device="cuda")
    call = m.spmspv if layout == celty.LAYOUT_COLUMN else m.spmspv_static
    xd = torch.zeros(K, dtype=torch.float16, device="cuda")
    ys = [torch.full((M,), 3.0, device="cuda") for _ in range(3)]
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        call(xd, 1.0, y=ys[0])
    side.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for y in ys:
            call(xd, 1.0, y=y)
    for seed in range(4):
        x = synth.integer_activations(90 + seed, K)
        xd.copy_(torch.from_numpy(x))
        for y in ys:
            y.fill_(float(seed - 7))
        graph.replay()
        torch.cuda.synchronize()
        y_ref, _ = orc.masked_gemv(W, mask, x, 1.0, threads=4)
        for y in ys:
            assert np.array_equal(y.cpu().numpy().astype(np.float64), y_ref)
