"""Products of layers whose thread blocks own few columns, dealt to them whatever x is, against the oracle and against the
kernel that ranks the survivors (variant 256): the edges of 32, 64, 96 and 128 columns per block, row parts of unequal block
counts, more blocks than columns, survivors that cluster in x."""
import threading

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


def test_the_binding_takes_and_refuses_what_it_should():
    """Calls through the native module: the caller's y comes back itself, a made one is new; wrong types, sizes and strides
    are refused before anything is launched, and the library's own refusals carry its status."""
    M, K = 64, 48
    W = synth.integer_weights(3, M, K)
    m = celty.Matrix(W, None, device="cuda")
    x = torch.from_numpy(synth.integer_activations(4, K)).cuda()
    y = torch.full((M,), 9.0, device="cuda")
    y_ref, _ = orc.masked_gemv(W, np.ones((M, K), np.uint8), x.cpu().numpy(), 1.0, threads=1)
    assert m.spmspv(x, 1, y=y) is y and m.spmspv(x, np.float32(1.0)) is not y
    assert np.array_equal(y.cpu().numpy().astype(np.float64), y_ref)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    z = m.spmspv(x, 1.0, y=torch.zeros(M, device="cuda"), stream=side)
    side.synchronize()
    assert torch.equal(z, y)
    for bad in (x.float(), x[:-1], torch.zeros(2 * K, dtype=torch.float16, device="cuda")[::2]):
        for call in (m.spmspv, m.spmspv_ex, m.spmspv_static):
            with pytest.raises(AssertionError):
                call(bad, 1.0)
    for bad in (y.half(), y[:-1], torch.zeros(2 * M, device="cuda")[::2]):
        with pytest.raises(AssertionError):
            m.spmspv(x, 1.0, y=bad)
    with pytest.raises(AssertionError):
        m.spmspv_ex(x, 1.0, fp16_out=torch.zeros(M, device="cuda"))
    with pytest.raises(AssertionError):
        m.spmspv_list(x, x, x)
    with pytest.raises(AssertionError):
        m.spmspv_batch(x, 1.0)
    with pytest.raises(TypeError):
        m.spmspv(x.cpu().numpy(), 1.0)
    for tau in (-1.0, float("nan"), 1e300):
        with pytest.raises(celty.CeltyError) as e:
            m.spmspv(x, tau)
        assert e.value.status == -1
    torch.cuda.synchronize()


# 4096 columns in two row parts of 74 blocks (56 columns each), 8192 (111 each)
@pytest.mark.parametrize("M,K", [(4096, 4096), (3000, 8192)])
def test_survivors_that_lie_together_in_x(M, K):
    """Zeroed heads of 64 and 128 activations, half of every head, and one stretch of x: such survivors are dealt to blocks
    as unevenly as the rule allows (a call's values do not depend on it)."""
    W = synth.integer_weights(7, M, K)
    mask = synth.mask_bernoulli(7, M, K, 0.5)
    m = celty.Matrix(W, mask, tile_rows=64 if M == 4096 else 48, device="cuda")
    rng = np.random.default_rng(K)
    i = np.arange(K)
    heads = rng.random(K // 128) < 0.5
    for keep in (heads[i // 128], (i // 64) % 2 == 0, i % 128 < 64, i < K // 8, i >= K - 40, i % 148 < 2):
        x = np.where(keep, rng.integers(1, 4, K) * rng.choice([-1, 1], K), 0).astype(np.float16)
        y_ref, _ = orc.masked_gemv(W, mask, x, 0.5, threads=8)
        xd = torch.from_numpy(x).cuda()
        for y in (m.spmspv(xd, 0.5, y=torch.full((M,), 5.0, device="cuda")), m.spmspv_static(xd, 0.5)):
            assert np.array_equal(y.cpu().numpy().astype(np.float64), y_ref)
        m.spmspv(xd, 0.5)
        gi, gv = m.last_compaction()
        oi, ov, _ = orc.compact(x, 0.5)
        assert np.array_equal(gi.cpu().numpy(), oi) and np.array_equal(gv.cpu().numpy().view(np.uint16), ov)
        assert m.last_status() == 0


def test_no_call_takes_a_vector_that_is_too_short_or_elsewhere():
    """The library gets bare pointers: sizes, types, strides and memory are the binding's to check, in every call.  Longer
    vectors are taken where only their beginning is written or read, and so is page-locked host memory."""
    M, K = 64, 48
    W = synth.integer_weights(5, M, K)
    m = celty.Matrix(W, None, device="cuda")
    half, dev = torch.float16, "cuda"
    x = torch.from_numpy(synth.integer_activations(6, K)).cuda()
    gate_up = torch.randn(2 * K, device=dev)

    def short(t):
        return (t[:-1], t.repeat(2)[::2], t.cpu(), t.double())

    y, f, h = torch.zeros(M, device=dev), torch.zeros(M, dtype=half, device=dev), torch.zeros(K, dtype=half, device=dev)
    for bad in short(y):
        for call in (lambda: m.spmspv(x, 1.0, y=bad), lambda: m.spmspv_ex(x, 1.0, y=bad), lambda: m.spmspv_static(x, 1.0, y=bad),
                     lambda: m.spmspv_swiglu(gate_up, 1.0, y=bad), lambda: m.spmspv_batch(x[None], 1.0, y=bad[None])):
            with pytest.raises(AssertionError):
                call()
    for bad in short(f):
        for call in (lambda: m.spmspv_ex(x, 1.0, fp16_out=bad), lambda: m.spmspv_swiglu(gate_up, 1.0, fp16_out=bad)):
            with pytest.raises(AssertionError):
                call()
    for bad in short(h):
        with pytest.raises(AssertionError):
            m.spmspv_swiglu(gate_up, 1.0, h_out=bad)
    for bad in short(gate_up):
        with pytest.raises(AssertionError):
            m.spmspv_swiglu(bad, 1.0)
    mid = celty.SwigluOut(M // 2, 0.1, dev)
    for name in ("h", "idx", "val", "count"):
        good = getattr(mid, name)
        for bad in (good[:-1], good.cpu(), good.double()) + ((good.repeat(2)[::2],) if name != "count" else ()):
            setattr(mid, name, bad)
            with pytest.raises(AssertionError):
                m.spmspv_ex(x, 1.0, swiglu=mid)
        setattr(mid, name, good)
    idx, val = (x.abs() > 1).nonzero().flatten().int(), x[x.abs() > 1]
    n = torch.tensor([idx.numel()], dtype=torch.int32, device=dev)
    for bad in (dict(y=y[:-1]), dict(y=y.cpu()), dict(y=y.half()), dict(idx=idx.cpu()), dict(idx=idx.repeat(2)[::2]), dict(idx=idx.long()),
                dict(val=val.cpu()), dict(val=val.repeat(2)[::2]), dict(val=val.float()), dict(count=n[:0]), dict(count=n.cpu()),
                dict(fp16_out=f[:-1]), dict(fp16_out=f.repeat(2)[::2])):
        with pytest.raises(AssertionError):
            m.spmspv_list(**{**dict(idx=idx, val=val, count=n), **bad})

    # what is longer than it has to be, or page-locked, is taken
    want = m.spmspv(x, 1.0)
    wide, wide_h = torch.full((M + 9,), 3.0, device=dev), torch.full((K + 9,), 3.0, dtype=half, device=dev)
    assert m.spmspv_list(idx, val.view(torch.int16), n, y=wide) is wide and torch.equal(wide[:M], want) and torch.all(wide[M:] == 3)
    longer = celty.SwigluOut(M, 0.1, dev)
    assert torch.equal(m.spmspv_ex(x, 1.0, swiglu=longer), want)
    plain = m.spmspv_swiglu(gate_up, 1.0)
    again = m.spmspv_swiglu(gate_up, 1.0, y=wide, h_out=wide_h)[:M]
    apart = torch.from_numpy(np.abs(W).astype(np.float32)).cuda() @ wide_h[:K].float().abs() * (2 * K * 2.0 ** -24)
    assert torch.all((again - plain).abs() <= apart) and torch.all(wide_h[K:] == 3)      # K FP32 additions in another order
    pinned = x.cpu().pin_memory()
    assert torch.equal(m.spmspv(pinned, 1.0, y=y), want)
    with pytest.raises(AssertionError):
        m.spmspv(pinned, 1.0)                                     # y would be made in pageable memory
    assert m.last_status() == 0


def test_first_calls_of_several_threads_on_one_handle():
    """A handle's launches are worked out by the first call of each kind: threads whose first calls meet (on one stream, which
    keeps their kernels apart) all launch the finished plan."""
    M, K, threads = 640, 512, 6
    W = synth.integer_weights(8, M, K)
    mask = synth.mask_bernoulli(8, M, K, 0.5)
    first = celty.Matrix(W, mask, device="cuda")
    X = np.stack([synth.integer_activations(70 + n, K) for n in range(threads)])
    ref = np.stack([orc.masked_gemv(W, mask, X[n], 1.0, threads=4)[0] for n in range(threads)])
    xd = torch.from_numpy(X).cuda()
    lists = [(torch.from_numpy(i).cuda(), torch.from_numpy(v.view(np.int16)).cuda(), torch.tensor([i.size], dtype=torch.int32, device="cuda"))
             for i, v, _ in (orc.compact(X[n], 1.0) for n in range(threads))]
    torch.cuda.synchronize()
    for _ in range(12):
        m = first.clone("cuda")
        ys, failed, start = [None] * threads, [], threading.Barrier(threads)

        def work(n):
            try:
                start.wait()
                calls = [lambda: m.spmspv(xd[n], 1.0), lambda: m.spmspv_list(*lists[n]), lambda: m.spmspv_batch(xd[:2], 1.0)]
                ys[n] = [calls[(n + k) % 3]() for k in range(3)], [(n + k) % 3 for k in range(3)]
            except BaseException as e:                            # noqa: BLE001
                failed.append(e)

        workers = [threading.Thread(target=work, args=(n,)) for n in range(threads)]
        for w in workers:
            w.start()
        for w in workers:
            w.join()
        assert not failed
        assert m.last_status() == 0
        for n in range(threads):
            for y, kind in zip(*ys[n]):
                want = ref[:2] if kind == 2 else ref[n]
                assert np.array_equal(y.cpu().numpy().astype(np.float64), want), (n, kind)


def test_the_plan_names_the_kernel():
    """At most 512 columns per block (384 where blocks left over can be shared, 20 000 / rows per lane for several vectors): dealt;
    more, several slabs per block, or on request: ranked.  A list is shared by the
    kernel that deals unless left-over blocks serve several row parts.  A caller of the C entry with room for ten words
    gets ten."""
    def plan(M, K, variant=0, **kw):
        m = celty.Matrix(synth.integer_weights(1, M, K), None, device="cuda", **kw)
        m.set_launch(variant=variant)
        p = m.launch_plan()
        assert 148 // p["row_parts"] == p["grid"] // p["row_parts"]                # one block per SM of a B200
        return p

    ranked, direct = "k_spmspv_fused", "k_spmspv_direct"
    for K, kernel in ((148 * 128, direct), (148 * 128 + 1, direct), (148 * 512, direct), (148 * 512 + 1, ranked)):
        p = plan(40, K)
        assert (p["kernel"], p["list_kernel"]) == (kernel, direct)
    for K, kernel in ((18 * 384, direct), (18 * 384 + 1, ranked)):                 # eight row parts, four blocks left over
        p = plan(256, K, tile_rows=1)
        assert (p["kernel"], p["row_parts"], p["parts_per_spare_block"]) == (kernel, 8, 1 if kernel == direct else 2)
    for N in range(2, 9):
        for M, rows, most in ((40, 0, 512), (4096, 128, 156)):
            columns = most * (148 // N)
            for K, kernel in ((columns, direct), (columns + 1, ranked)):
                assert plan(M, K, tile_rows=rows)["batch_kernels"][N] == kernel, (N, K)
    for variant in (2, 128, 256):
        p = plan(300, 400, variant)
        assert p["kernel"] == ranked and p["list_kernel"] in (ranked, None)
    assert plan(300, 400, tile_rows=2, slabs_per_block=2)["kernel"] == ranked
    m = celty.Matrix(synth.integer_weights(1, 40, 40), None, device="cuda")
    import ctypes
    out = (ctypes.c_int32 * 20)(*[-7] * 20)
    for n in (10, 11, 12, 18, 19, 20):
        assert celty.load().celty_launch_plan(m._h, out, n) == 0
        assert out[min(n, 19):] == [-7] * (20 - min(n, 19)) and out[0] == 148
    assert celty.load().celty_launch_plan(m._h, out, 9) == -1


def test_the_tables_leave_room_for_eight_teams():
    """A block's accumulators and ring slots fill shared memory nearly to the brim on this layer (128 rows per lane, one row
    part): what the kernel keeps per column may not cost it a team."""
    M, K = 4096, 11008
    W = synth.weights(9, M, K)
    plan = celty.Matrix(W, synth.mask_magnitude(W, 0.5), device="cuda").launch_plan()
    assert plan["kernel"] == "k_spmspv_direct" and plan["row_parts"] == 1
    assert plan["teams_per_slab"] == 8 and plan["warp_pairs"] == 1
