"""Images that go to the GPU through the library's page-locked memory arrive whole: sizes around the pieces they are cut into,
several threads and streams at once, memory given back in between."""
import threading

import numpy as np
import pytest
import torch

from paper_2608_01536_b200 import build, celty, synth

pytestmark = pytest.mark.gpu

PIECE = 512 << 10


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    assert torch.cuda.is_available(), "these tests need a CUDA device"
    celty.load()


def _matrix(bytes_wanted, seed):
    M = 64                                                        # dense columns: 48 + 32 * 20 bytes and their offset
    K = max(1, bytes_wanted // 692)
    return celty.Matrix(synth.integer_weights(seed, M, K), np.ones((M, K), np.uint8))


@pytest.mark.parametrize("size", [1000, PIECE - 4096, PIECE, PIECE + 4096, 3 * PIECE, 3 * PIECE + 1, 40 * PIECE + 77])
def test_an_uploaded_image_is_the_packed_one(size):
    m = _matrix(size, size % 97)
    for _ in range(2):
        m.to("cuda")
        assert np.array_equal(m._image.cpu().numpy(), m.host_image()[0])
        celty.release_staging()


def test_uploads_of_several_threads_and_streams():
    ms = [_matrix(9 * PIECE + 1000 * k, k) for k in range(4)]
    bad = []

    def work(m):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                for _ in range(5):
                    m.to("cuda", stream=s)
                    if not np.array_equal(m._image.cpu().numpy(), m.host_image()[0]):
                        bad.append("differs")
        except BaseException as e:                                # noqa: BLE001
            bad.append(e)

    threads = [threading.Thread(target=work, args=(m,)) for m in ms]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    celty.release_staging()
    assert not bad


def test_an_upload_beside_another_threads_capture():
    """A capture that watches all threads goes on while another thread takes the page-locked memory and uploads."""
    celty.release_staging()
    m, small = _matrix(6 * PIECE, 3), celty.Matrix(synth.integer_weights(1, 64, 64), device="cuda")
    x = torch.ones(64, dtype=torch.float16, device="cuda")
    small.spmspv(x, 0.5)
    buffers = [torch.empty(b, dtype=torch.uint8, device="cuda") for b in m.device_bytes()]
    stream, bad = torch.cuda.Stream(), []
    torch.cuda.synchronize()

    def work():
        try:
            torch.cuda.set_device(0)
            celty._check(celty.load().celty_bind_device(m._h, buffers[0].data_ptr(), buffers[0].numel(), buffers[1].data_ptr(),
                                                        buffers[1].numel(), stream.cuda_stream), "celty_bind_device")
        except BaseException as e:                                # noqa: BLE001
            bad.append(e)

    y = torch.empty(64, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        small.spmspv(x, 0.5, y=y)
        t = threading.Thread(target=work)
        t.start()
        t.join()
    graph.replay()
    torch.cuda.synchronize()
    assert not bad
    assert np.array_equal(buffers[0].cpu().numpy(), m.host_image()[0])
    assert np.array_equal(y.cpu().numpy(), small.spmspv(x, 0.5).cpu().numpy())


def test_an_upload_on_the_threads_own_stream():
    """cudaStreamPerThread (handle 2) means the calling thread's stream: reads enqueued there behind each of several uploads into one
    buffer find the image that was uploaded last."""
    ms = [_matrix(40 * PIECE, k) for k in range(2)]
    assert ms[0].device_bytes() == ms[1].device_bytes()
    image, ws = [torch.empty(b, dtype=torch.uint8, device="cuda") for b in ms[0].device_bytes()]
    torch.cuda.synchronize()
    stream, read = torch.cuda.ExternalStream(2), []
    for k in range(6):
        m = ms[k % 2]
        celty._check(celty.load().celty_bind_device(m._h, image.data_ptr(), image.numel(), ws.data_ptr(), ws.numel(), 2), "celty_bind_device")
        with torch.cuda.stream(stream):
            read.append(torch.empty(image.numel(), dtype=torch.uint8, pin_memory=True))
            read[-1].copy_(image, non_blocking=True)
    stream.synchronize()
    for k in range(6):
        assert np.array_equal(read[k].numpy(), ms[k % 2].host_image()[0]), k


@pytest.mark.parametrize("size", [2 * PIECE, 20 * PIECE])
def test_an_upload_behind_work_of_its_stream(size):
    """The image of before is read by work that the stream has yet to do when the next one is bound to the same memory."""
    a, b = _matrix(size, 1), _matrix(size, 2)
    assert a.device_bytes() == b.device_bytes()
    image, ws = [torch.empty(n, dtype=torch.uint8, device="cuda") for n in a.device_bytes()]
    torch.cuda.synchronize()
    stream, read = torch.cuda.Stream(), []
    with torch.cuda.stream(stream):
        for m in (a, b, a):
            celty._check(celty.load().celty_bind_device(m._h, image.data_ptr(), image.numel(), ws.data_ptr(), ws.numel(), stream.cuda_stream), "celty_bind_device")
            torch.cuda._sleep(20_000_000)                         # some 10 ms
            read.append(image.clone())
    stream.synchronize()
    for m, r in zip((a, b, a), read):
        assert np.array_equal(r.cpu().numpy(), m.host_image()[0])
