import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA device (run on a B200)")


def read_golden(name):
    """Parse tests/golden/<name>: '#' comments, 'case <id>' headers, 'key: v v v' lines."""
    cases, cur = {}, None
    with open(os.path.join(ROOT, "tests", "golden", name)) as f:
        for line in f:
            line = line.split("#", 1)[0].strip()
            if not line:
                continue
            if line.startswith("case "):
                cur = {}
                cases[line[5:].strip()] = cur
                continue
            key, _, rest = line.partition(":")
            cur[key.strip()] = [int(t) for t in rest.split()]
    return cases


@pytest.fixture(scope="session")
def golden():
    return read_golden


def lane_tile_rows(M, S, R, C):
    """Row of W behind (tile t = 32*s + L, local row i) for the LANE_TILE row map, written out from its
    definition in the public header; -1 where that row does not exist.  Shape (32*S, R)."""
    import numpy as np
    t = np.arange(32 * S)[:, None]
    i = np.arange(R)[None, :]
    s, L = t // 32, t % 32
    rows = (((i // C) * S + s) * C + i % C) * 32 + L
    return np.where(rows < M, rows, -1)


def permute_for_lane_tiles(W, mask, S, R, C):
    """(W', mask', rows): the matrix whose consecutive tiles of R rows are the library's lane tiles, so
    that the oracle's encoder with tile_rows=R sees what the library stores; rows[p] = row of W at p."""
    import numpy as np
    M, K = W.shape
    rows = lane_tile_rows(M, S, R, C).reshape(-1)
    live = rows >= 0
    assert np.array_equal(np.sort(rows[live]), np.arange(M))         # a permutation of the rows
    if mask is None:
        mask = ((W.view(np.uint16) & 0x7FFF) != 0).astype(np.uint8)
    Wp = np.zeros((rows.size, K), W.dtype)
    mp = np.zeros((rows.size, K), np.uint8)
    Wp[live] = W[rows[live]]
    mp[live] = mask[rows[live]]
    return Wp, mp, rows


def hold_some_sms(celty, synth, stream, blocks=40, polls=400_000):
    """Enqueues on `stream` a product that keeps `blocks - 1` SMs to itself for some tenths of a second, by a bounded
    wait that runs out: its ticket is moved so that all blocks but one wait for a count that never comes.  Returns the
    handle (whose next last_status() is CELTY_ETIMEOUT) and an event behind the call."""
    import time

    import torch
    holder = celty.Matrix(synth.weights(70, 4096, 1024), None, device="cuda")
    holder.set_launch(grid=blocks)
    plan = holder.launch_plan()
    assert plan["grid"] == blocks and plan["smem_bytes"] > 120 * 1024        # no block of the products fits beside one
    x = torch.from_numpy(synth.activations(71, 1024, "laplace")).cuda()
    holder.spmspv(x, 0.5)
    torch.cuda.synchronize()
    assert holder.last_status() == 0
    ticket = holder._ws[8:12].view(torch.int32)
    ticket[0] = blocks - 1
    holder.set_wait_limit(polls)
    torch.cuda.synchronize()
    done = torch.cuda.Event()
    holder.spmspv(x, 0.5, stream=stream)
    done.record(stream)
    time.sleep(0.01)                                                         # it is on the SMs now
    return holder, done
