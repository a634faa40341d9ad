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
