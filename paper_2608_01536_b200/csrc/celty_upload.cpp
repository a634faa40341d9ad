// Host-to-device copies of images through page-locked memory.  A copy from pageable memory is one host thread's in the driver, 4
// GB/s; here up to kUploadThreads threads copy pieces into slots of page-locked memory, and one of them, the caller's, enqueues the copies
// from there.  It alone makes CUDA calls: a stream handle may mean another stream in another thread (cudaStreamPerThread), and the
// caller's context need not be the one that cudaSetDevice would make current.  The 8 MB are taken by the first upload, used by one upload at a
// time and given back by celty_release_staging.  An upload ends when its copies have left the slots, so that it waits for no other stream's
// work, nor leaves events for another context.
#include "celty_upload.h"

#include <algorithm>
#include <condition_variable>
#include <cstring>
#include <exception>
#include <mutex>
#include <thread>
#include <vector>

#include "celty_internal.h"

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
struct Staging {
    std::mutex mu;
    Raw<uint8_t> memory;

    // The slots, page-locked; null: not to be had (mu is held).
    uint8_t *slots()
    {
        try {
            if (memory.size() == 0) memory.allocate(kUploadSlots * kUploadPiece);
        } catch (const std::exception &) {
            return nullptr;
        }
        cudaPointerAttributes is{};
        if (cudaPointerGetAttributes(&is, memory.data()) == cudaSuccess && is.type == cudaMemoryTypeHost) return memory.data();
        (void)cudaGetLastError();
        if (cudaHostRegister(memory.data(), memory.size(), cudaHostRegisterPortable) == cudaSuccess) return memory.data();
        (void)cudaGetLastError();
        return nullptr;
    }
};

Staging &staging()
{
    static Staging *s = new Staging;                              // (never destroyed: the runtime may be gone by then)
    return *s;
}

// The pieces of an image on their way through the slots, piece i through slot i mod kUploadSlots.
class Pieces {
public:
    Pieces(uint8_t *slots, const uint8_t *from, size_t bytes) : slots_(slots), from_(from), bytes_(bytes) {}
    int64_t count() const { return (int64_t)((bytes_ + kUploadPiece - 1) / kUploadPiece); }
    size_t size(int64_t i) const { return std::min(kUploadPiece, bytes_ - (size_t)i * kUploadPiece); }
    uint8_t *slot(int64_t i) const { return slots_ + (size_t)(i % kUploadSlots) * kUploadPiece; }

    // A thread that fills slots: the next pieces, each as soon as its slot is free.
    void fill_all()
    {
        std::unique_lock<std::mutex> lock(mu_);
        while (!stopped_ && claimed_ < count()) {
            const int64_t i = claimed_++;
            changed_.wait(lock, [&] { return stopped_ || i < copied_ + kUploadSlots; });
            if (stopped_) return;
            fill(i, lock);
        }
    }

    // Returns when piece i is there; fills others, or i itself, meanwhile.
    void wait_filled(int64_t i)
    {
        std::unique_lock<std::mutex> lock(mu_);
        while (filled_[i % kUploadSlots] != i + 1) {
            if (claimed_ < std::min(count(), copied_ + kUploadSlots)) fill(claimed_++, lock);
            else changed_.wait(lock);
        }
    }

    // The copies of the first n pieces have been made: their slots are free.
    void copied(int64_t n)
    {
        std::lock_guard<std::mutex> lock(mu_);
        copied_ = n;
        changed_.notify_all();
    }

    void stop()
    {
        std::lock_guard<std::mutex> lock(mu_);
        stopped_ = true;
        changed_.notify_all();
    }

private:
    void fill(int64_t i, std::unique_lock<std::mutex> &lock)
    {
        lock.unlock();
        std::memcpy(slot(i), from_ + (size_t)i * kUploadPiece, size(i));
        lock.lock();
        filled_[i % kUploadSlots] = i + 1;
        changed_.notify_all();
    }

    uint8_t *const slots_;
    const uint8_t *const from_;
    const size_t bytes_;
    std::mutex mu_;
    std::condition_variable changed_;
    int64_t claimed_ = 0, copied_ = 0;
    int64_t filled_[kUploadSlots] = {};                           // i + 1 when piece i is there
    bool stopped_ = false;
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
    Staging &stage = staging();
    std::unique_lock<std::mutex> lock(stage.mu, std::defer_lock);
    bool staged = capturing == cudaStreamCaptureStatusNone && bytes >= kUploadPiece && lock.try_lock();
    if (staged && cudaStreamQuery(st) != cudaSuccess) {
        (void)cudaGetLastError();
        lock.unlock();
        staged = false;
    }
    uint8_t *const slots = staged ? stage.slots() : nullptr;
    // (first, and waited for with the copies: the next layer's upload finds the stream idle)
    if ((err = cudaMemsetAsync(clear, 0, clear_bytes, st)) != cudaSuccess) return err;
    if (!slots) return cudaMemcpyAsync(to, from, bytes, cudaMemcpyHostToDevice, st);
    Pieces pieces(slots, from, bytes);
    std::vector<std::thread> threads;
    try {
        const int64_t want = std::min<int64_t>({kUploadThreads, (pieces.count() + 2) / 3, std::max(1u, std::thread::hardware_concurrency())});
        threads.reserve((size_t)want);
        for (int64_t t = 1; t < want; ++t) threads.emplace_back([&] { pieces.fill_all(); });
    } catch (const std::exception &) {                            // no (more) threads to be had: those there are do it
    }
    cudaEvent_t done[kUploadSlots] = {};                          // of a slot's last copy
    cudaEvent_t last = nullptr;
    for (int64_t i = 0, made = 0; i < pieces.count(); ++i) {
        for (; made < i; ++made) {
            const cudaEvent_t e = done[made % kUploadSlots];
            err = i - made == kUploadSlots ? cudaEventSynchronize(e) : cudaEventQuery(e);
            if (err != cudaSuccess) break;
        }
        if (err == cudaErrorNotReady) (void)cudaGetLastError();
        else if (err != cudaSuccess) break;
        pieces.copied(made);
        pieces.wait_filled(i);
        cudaEvent_t &e = done[i % kUploadSlots];
        if (!e && (err = cudaEventCreateWithFlags(&e, cudaEventDisableTiming)) != cudaSuccess) break;
        err = cudaMemcpyAsync(static_cast<uint8_t *>(to) + (size_t)i * kUploadPiece, pieces.slot(i), pieces.size(i), cudaMemcpyHostToDevice, st);
        if (err == cudaSuccess) err = cudaEventRecord(e, st);
        if (err != cudaSuccess) break;
        last = e;
    }
    pieces.stop();
    for (std::thread &t : threads) t.join();
    if (last) {
        const cudaError_t waited = cudaEventSynchronize(last);
        if (err == cudaSuccess) err = waited;
    }
    for (cudaEvent_t e : done)
        if (e) cudaEventDestroy(e);
    return err;
}

cudaError_t release_staging()
{
    RelaxedCapture relaxed;
    Staging &stage = staging();
    std::lock_guard<std::mutex> lock(stage.mu);
    if (stage.memory.size() == 0) return cudaSuccess;
    cudaError_t err = cudaHostUnregister(stage.memory.data());
    if (err == cudaErrorHostMemoryNotRegistered) {
        (void)cudaGetLastError();
        err = cudaSuccess;
    }
    if (err == cudaSuccess) stage.memory.reset();
    return err;
}

}  // namespace celty
