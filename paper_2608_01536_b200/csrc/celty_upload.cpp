// Host-to-device copies of images through page-locked memory.  A copy from pageable memory is one host thread's in the driver, 4
// GB/s; here up to kUploadThreads threads copy pieces into slots of page-locked memory, and one of them, the caller's, enqueues the copies
// from there.  It alone makes CUDA calls: a stream handle may mean another stream in another thread (cudaStreamPerThread), and the
// caller's context need not be the one that cudaSetDevice would make current.  The 8 MB are taken by the first upload, used by one upload at a
// time and given back by celty_release_staging.  An upload ends when its copies have left the slots, so that it waits for no other stream's
// work, nor leaves events for another context.  celty_bind_device with a new image, from pageable memory / this way: 6.3 MB 1.5 / 1.1 ms, 12.6 MB
// 2.5 / 1.2, 57 MB 6.5 / 2.6, 171 MB 16.5 / 6.3.  Bound by the threads' start, then by their copies.
#include "celty_upload.h"

#include <algorithm>
#include <atomic>
#include <cstring>
#include <exception>
#include <mutex>
#include <thread>
#include <type_traits>
#include <vector>

#include <sys/mman.h>

#include "celty_signal.h"

namespace celty {

namespace {

constexpr int kUploadThreads = 8, kUploadSlots = 16;
constexpr size_t kUploadPiece = (size_t)512 << 10;

// Another thread's stream capture (of the mode that watches all threads) does not mind this thread's allocations and waits.
struct RelaxedCapture {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

// Ordinary memory that is registered: cudaDeviceReset, or the end of the context that was current, ends the registration and not the memory.
// (Not of the heap, whose largest blocks it would lie between.)
struct Staging {
    static constexpr size_t bytes = kUploadSlots * kUploadPiece;
    std::mutex mu;
    uint8_t *memory = nullptr;

    // The slots, page-locked; null: not to be had (mu is held).
    uint8_t *slots()
    {
        if (!memory) {
            void *const m = mmap(nullptr, bytes, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
            if (m == MAP_FAILED) return nullptr;
            memory = static_cast<uint8_t *>(m);
        }
        cudaPointerAttributes is{};
        if (cudaPointerGetAttributes(&is, memory) == cudaSuccess && is.type == cudaMemoryTypeHost) return memory;
        (void)cudaGetLastError();
        if (cudaHostRegister(memory, bytes, cudaHostRegisterPortable) == cudaSuccess) return memory;
        (void)cudaGetLastError();
        return nullptr;
    }
};

Staging stage;
static_assert(std::is_trivially_destructible<Staging>::value, "at the process's end the runtime may be gone");

// The pieces of an image on their way through the slots, piece i through slot i mod kUploadSlots.
class Pieces {
public:
    Pieces(uint8_t *slots, const uint8_t *from, size_t bytes)
        : slots_(slots), from_(from), bytes_(bytes), count_((int64_t)((bytes + kUploadPiece - 1) / kUploadPiece)) {}
    int64_t count() const { return count_; }
    uint8_t *slot(int64_t i) const { return slots_ + (size_t)(i % kUploadSlots) * kUploadPiece; }
    size_t size(int64_t i, int64_t n) const { return std::min((size_t)n * kUploadPiece, bytes_ - (size_t)i * kUploadPiece); }      // of n pieces from i on
    bool filled(int64_t i) const { return filled_[i % kUploadSlots] == i + 1; }

    // A thread that fills slots: the next pieces, each as soon as its slot is free.
    void fill_all()
    {
        while (!stopped_ && claimed_ < count_)
            if (!fill_next()) free_.wait([&] { return stopped_ || claimed_ >= count_ || claimed_ < copied_ + kUploadSlots; });
    }

    // Returns when piece i is there; fills others, or i itself, meanwhile.
    void wait_filled(int64_t i)
    {
        while (!filled(i))
            if (!fill_next()) there_.wait([&] { return filled(i); });
    }

    // The copies of the first n pieces have been made: their slots are free.
    void copied(int64_t n)
    {
        copied_ = n;
        free_.raise();
    }

    void stop()
    {
        stopped_ = true;
        free_.raise();
    }

private:
    bool fill_next()                                              // false: no piece whose slot is free is left
    {
        int64_t i = claimed_;
        do {
            if (i >= std::min<int64_t>(count_, copied_ + kUploadSlots)) return false;
        } while (!claimed_.compare_exchange_weak(i, i + 1));
        std::memcpy(slot(i), from_ + (size_t)i * kUploadPiece, size(i, 1));
        filled_[i % kUploadSlots] = i + 1;
        there_.raise();
        return true;
    }

    uint8_t *const slots_;
    const uint8_t *const from_;
    const size_t bytes_;
    const int64_t count_;
    std::atomic<int64_t> claimed_{0}, copied_{0};
    std::atomic<int64_t> filled_[kUploadSlots] = {};              // i + 1 when piece i is there
    std::atomic<bool> stopped_{false};
    Signal there_, free_;
};

}  // namespace

// The pageable way go what a stream capture would have to replay, small images, those that come while the staging memory is in use, and
// those behind work that their stream has not done yet: the wait for the copies would be one for that work.
cudaError_t upload(void *to, const uint8_t *from, size_t bytes, void *clear, size_t clear_bytes, cudaStream_t st)
{
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusActive;
    cudaError_t err = cudaStreamIsCapturing(st, &capturing);
    if (err != cudaSuccess) return err;
    RelaxedCapture relaxed;
    std::unique_lock<std::mutex> lock(stage.mu, std::defer_lock);
    bool staged = capturing == cudaStreamCaptureStatusNone && bytes >= kUploadPiece && lock.try_lock();
    if (staged && cudaStreamQuery(st) != cudaSuccess) {
        (void)cudaGetLastError();
        lock.unlock();
        staged = false;
    }
    uint8_t *const slots = staged ? stage.slots() : nullptr;
    if (!slots) {
        err = cudaMemcpyAsync(to, from, bytes, cudaMemcpyHostToDevice, st);
        return err == cudaSuccess ? cudaMemsetAsync(clear, 0, clear_bytes, st) : err;
    }
    Pieces pieces(slots, from, bytes);
    std::vector<std::thread> threads;
    try {
        const int64_t want = std::min<int64_t>({kUploadThreads, (pieces.count() + 2) / 3, std::max(1u, std::thread::hardware_concurrency())});
        threads.reserve((size_t)want);
        for (int64_t t = 1; t < want; ++t) threads.emplace_back([&] { pieces.fill_all(); });
    } catch (const std::exception &) {                            // no (more) threads to be had: those there are do it
    }
    // The pieces that are there are copied together, up to the end of their quarter of the slots, and a quarter is free again behind its event.
    constexpr int quarter = kUploadSlots / 4;
    cudaEvent_t done[4] = {};
    int64_t made = 0, recorded = 0;                               // quarters copied, quarters with an event behind them
    for (int64_t i = 0, n; i < pieces.count(); i += n) {
        for (; made < recorded; ++made) {
            const cudaEvent_t e = done[made % 4];
            err = i == (made + 4) * quarter ? cudaEventSynchronize(e) : cudaEventQuery(e);
            if (err != cudaSuccess) break;
        }
        if (err == cudaErrorNotReady) (void)cudaGetLastError();
        else if (err != cudaSuccess) break;
        pieces.copied(made * quarter);
        pieces.wait_filled(i);
        const int64_t end = std::min(pieces.count(), (i / quarter + 1) * quarter);
        for (n = 1; i + n < end && pieces.filled(i + n); ++n) {}
        err = cudaMemcpyAsync(static_cast<uint8_t *>(to) + (size_t)i * kUploadPiece, pieces.slot(i), pieces.size(i, n), cudaMemcpyHostToDevice, st);
        if (err != cudaSuccess) break;
        if (i + n < end) continue;
        cudaEvent_t &e = done[recorded % 4];
        if (!e && (err = cudaEventCreateWithFlags(&e, cudaEventDisableTiming)) != cudaSuccess) break;
        if ((err = cudaEventRecord(e, st)) != cudaSuccess) break;
        ++recorded;
    }
    pieces.stop();
    for (std::thread &t : threads) t.join();
    // (the clearing is waited for as well: the next layer's upload finds the stream idle)
    if (err == cudaSuccess && (err = cudaMemsetAsync(clear, 0, clear_bytes, st)) == cudaSuccess) err = cudaEventRecord(done[0], st);
    if (err == cudaSuccess) err = cudaEventSynchronize(done[0]);
    else (void)cudaStreamSynchronize(st);                         // (there may be copies without an event)
    for (cudaEvent_t e : done)
        if (e) cudaEventDestroy(e);
    return err;
}

cudaError_t release_staging()
{
    RelaxedCapture relaxed;
    std::lock_guard<std::mutex> lock(stage.mu);
    if (!stage.memory) return cudaSuccess;
    cudaError_t err = cudaHostUnregister(stage.memory);
    if (err == cudaErrorHostMemoryNotRegistered) {
        (void)cudaGetLastError();
        err = cudaSuccess;
    }
    if (err != cudaSuccess) return err;
    munmap(stage.memory, Staging::bytes);
    stage.memory = nullptr;
    return cudaSuccess;
}

}  // namespace celty
