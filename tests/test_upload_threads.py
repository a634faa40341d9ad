"""Uploads of images against a CUDA runtime made of host code: a copy is made when something waits for it (or a query says it is
ready), and cudaStreamPerThread means a queue of the calling thread's own.  No GPU needed."""
import os
import subprocess

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2608_01536_b200", "csrc")
CUDA = os.path.join(os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"))), "include")

MAIN = r'''
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <deque>
#include <map>
#include <mutex>
#include <random>
#include <set>
#include <string>
#include <thread>
#include <vector>
#include <sys/mman.h>
#include "celty_upload.h"

// ---- the runtime: queues of copies and event marks
struct Op { void *to; const void *from; size_t n; std::vector<uint8_t> own; struct Event *mark; };
struct Event { bool ready = true; int polls = 0; std::string queue; };
std::recursive_mutex mu;
std::map<std::string, std::deque<Op>> queues;
std::map<std::string, int> calls;
std::set<std::thread::id> callers;
std::set<Event *> events;
struct Locked { size_t bytes; bool ours; };
std::map<uint8_t *, Locked> locked;
std::set<std::string> held;                      // queues that do not get on

std::string queue_of(cudaStream_t st)
{
    char name[64];
    snprintf(name, sizeof name, "%p", (void *)st);
    return st == cudaStreamPerThread ? std::to_string(std::hash<std::thread::id>()(std::this_thread::get_id())) : name;
}
void drain(const std::string &q, Event *up_to)
{
    auto &ops = queues[q];
    if (held.count(q)) { printf("a wait for the work of a queue that is held\n"); exit(3); }
    while (!ops.empty()) {
        Op op = std::move(ops.front());
        ops.pop_front();
        if (op.n) memcpy(op.to, op.own.empty() ? op.from : op.own.data(), op.n);
        if (op.mark) op.mark->ready = true;
        if (op.mark && op.mark == up_to) return;
    }
}
void called(const char *name) { ++calls[name]; callers.insert(std::this_thread::get_id()); }
#define CALL std::lock_guard<std::recursive_mutex> lock(mu); called(__func__)
extern "C" {
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) { CALL; *s = cudaStreamCaptureStatusNone; return cudaSuccess; }
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode *) { return cudaSuccess; }
cudaError_t cudaStreamQuery(cudaStream_t st) { CALL; return queues[queue_of(st)].empty() ? cudaSuccess : cudaErrorNotReady; }
cudaError_t cudaGetDevice(int *d) { CALL; *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { CALL; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned)
{
    CALL;
    *p = mmap(nullptr, n, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
    locked[(uint8_t *)*p] = Locked{n, true};
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) { CALL; munmap(p, locked.at((uint8_t *)p).bytes); locked.erase((uint8_t *)p); return cudaSuccess; }
cudaError_t cudaHostRegister(void *p, size_t n, unsigned)
{
    CALL;
    if (locked.count((uint8_t *)p)) return cudaErrorHostMemoryAlreadyRegistered;
    locked[(uint8_t *)p] = Locked{n, false};
    return cudaSuccess;
}
cudaError_t cudaHostUnregister(void *p) { CALL; return locked.erase((uint8_t *)p) ? cudaSuccess : cudaErrorHostMemoryNotRegistered; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) { CALL; a->type = locked.count((uint8_t *)p) ? cudaMemoryTypeHost : cudaMemoryTypeUnregistered; return cudaSuccess; }
void device_reset()                              // what was allocated page-locked is gone, what was registered is ordinary memory
{
    for (auto &l : locked) if (l.second.ours) munmap(l.first, l.second.bytes);
    locked.clear();
    events.clear();
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { CALL; Event *ev = new Event; events.insert(ev); *e = (cudaEvent_t)ev; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { CALL; events.erase((Event *)e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t st)
{
    CALL;
    Event *ev = (Event *)e;
    ev->ready = false; ev->polls = 0; ev->queue = queue_of(st);
    queues[ev->queue].push_back(Op{nullptr, nullptr, 0, {}, ev});
    return cudaSuccess;
}
cudaError_t cudaEventQuery(cudaEvent_t e)
{
    CALL;
    Event *ev = (Event *)e;
    if (!ev->ready && ++ev->polls >= 3 && !held.count(ev->queue)) drain(ev->queue, ev);
    return ev->ready ? cudaSuccess : cudaErrorNotReady;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e)
{
    CALL;
    Event *ev = (Event *)e;
    if (!ev->ready) drain(ev->queue, ev);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t st) { CALL; drain(queue_of(st), nullptr); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int c, size_t n, cudaStream_t st) { CALL; queues[queue_of(st)].push_back(Op{p, nullptr, n, std::vector<uint8_t>(n, (uint8_t)c), nullptr}); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *to, const void *from, size_t n, cudaMemcpyKind, cudaStream_t st)
{
    CALL;
    Op op{to, from, n, {}, nullptr};
    bool is_locked = false;
    for (auto &l : locked) is_locked |= (const uint8_t *)from >= l.first && (const uint8_t *)from < l.first + l.second.bytes;
    if (!is_locked) op.own.assign((const uint8_t *)from, (const uint8_t *)from + n);      // pageable: read before the call returns
    queues[queue_of(st)].push_back(std::move(op));
    return cudaSuccess;
}
}

uint8_t cleared[1000];
std::vector<uint8_t> image(size_t n, unsigned seed)
{
    std::vector<uint8_t> v(n);
    std::mt19937 r(seed);
    for (size_t i = 0; i + 4 <= n; i += 4) { const uint32_t w = r(); memcpy(&v[i], &w, 4); }
    return v;
}
#define CHECK(c) do { if (!(c)) { printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)

// A caller's stream: the image, others into the same place, and reads of it behind each copy, by the stream's order; the stream is busy
// with the read when the second one comes.
int ordered(cudaStream_t st, size_t n)
{
    std::vector<uint8_t> at(n), read[3];
    const std::string q = queue_of(st);
    for (int k = 0; k < 3; ++k) {
        const std::vector<uint8_t> from = image(n, (unsigned)(n + k));
        memset(cleared, 7, sizeof cleared);
        CHECK(celty::upload(at.data(), from.data(), n, cleared, sizeof cleared, st) == cudaSuccess);
        read[k].resize(n);
        { std::lock_guard<std::recursive_mutex> lock(mu); queues[q].push_back(Op{read[k].data(), at.data(), n, {}, nullptr}); }
        if (k != 0) { std::lock_guard<std::recursive_mutex> lock(mu); drain(q, nullptr); }
        if (k != 0) CHECK(cleared[0] == 0 && cleared[999] == 0);
    }
    { std::lock_guard<std::recursive_mutex> lock(mu); drain(q, nullptr); }
    for (int k = 0; k < 3; ++k) CHECK(read[k] == image(n, (unsigned)(n + k)));
    return 0;
}

int main(int, char **v)
{
    const std::string what = v[1];
    const cudaStream_t st = (cudaStream_t)atol(v[2]);
    const size_t n = (size_t)atol(v[3]);
    if (what == "ordered") {
        if (ordered(st, n)) return 1;
        CHECK(callers.size() == 1);              // of which a stream handle or a context may be the property
        CHECK(calls["cudaSetDevice"] == 0);
    }
    if (what == "held") {                        // a stream that does not get on holds up neither its own small uploads nor another's
        const cudaStream_t other = (cudaStream_t)77;
        std::vector<uint8_t> at(n), there(n), from = image(n, 1);
        CHECK(celty::upload(there.data(), from.data(), n, cleared, sizeof cleared, other) == cudaSuccess);
        const std::string q = queue_of(st);
        queues[q].push_back(Op{&at[0], from.data(), 1, {}, nullptr});
        held.insert(q);
        CHECK(celty::upload(at.data(), from.data(), n, cleared, sizeof cleared, st) == cudaSuccess);
        const std::vector<uint8_t> next = image(n, 2);
        CHECK(celty::upload(there.data(), next.data(), n, cleared, sizeof cleared, other) == cudaSuccess);
        drain(queue_of(other), nullptr);
        CHECK(there == next);
        held.clear();
        drain(q, nullptr);
        CHECK(at == from);
    }
    if (what == "reset") {                       // and one that is not followed by another upload
        if (ordered(st, n)) return 1;
        device_reset();
        if (ordered(st, n)) return 1;
        CHECK(n < (512 << 10) || locked.size() == 1);
        device_reset();
    }
    CHECK(events.empty());                       // (of the context that was current)
    CHECK(celty::release_staging() == cudaSuccess);
    CHECK(celty::release_staging() == cudaSuccess);
    return 0;
}
'''


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("upload")
    (d / "main.cpp").write_text(MAIN)
    exe = str(d / "upload")
    subprocess.check_call(["g++", "-O1", "-g", "-std=c++17", "-pthread", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-I", CUDA, os.path.join(CSRC, "celty_upload.cpp"),
                           str(d / "main.cpp"), "-o", exe])

    def run(*args):
        r = subprocess.run([exe, *map(str, args)], capture_output=True, text=True, timeout=120)
        assert r.returncode == 0, r.stdout + r.stderr
    return run


# handles 1 and 2 are cudaStreamLegacy and cudaStreamPerThread; sizes around the pieces of 512 KB, and beyond all slots
@pytest.mark.parametrize("stream", [0, 1, 2, 4096])
@pytest.mark.parametrize("size", [1000, (512 << 10) - 1, 512 << 10, (1536 << 10) + 1, 2 << 20, (8 << 20) - 1, (8 << 20) + 5, 20 << 20])
def test_an_upload_is_work_of_the_callers_stream(program, stream, size):
    program("ordered", stream, size)


@pytest.mark.parametrize("size", [1000, 512 << 10, 3 << 20, 8 << 20])
def test_an_upload_waits_for_no_other_work(program, size):
    program("held", 4096, size)


@pytest.mark.parametrize("size", [1000, 2 << 20, 20 << 20])
def test_uploads_go_on_after_a_device_reset(program, size):
    program("reset", 4096, size)
