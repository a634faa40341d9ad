// Waiting of host threads for one another (encoder, uploads).
#pragma once

#include <atomic>
#include <chrono>
#include <climits>
#include <cstdint>
#include <thread>

#include <linux/futex.h>
#include <sys/syscall.h>
#include <unistd.h>

namespace celty {

// What threads wait for lies in atomics of their own; a signal says that it may have changed.  Who waits looks for 0.2 ms, which most waits
// of an encoding or an upload do not take, and sleeps from then on: the processors may be wanted by other work, another layer's encoding
// perhaps.  All sleepers are woken at once.  (Asleep on a condition variable from 50 us on, 15 of them took its mutex one after the other:
// encoding 11008 x 4096 on 16 threads 9.5 ms instead of 7.4.)
class Signal {
public:
    // The caller has changed what others may wait for.
    void raise()
    {
        ++turn_;
        if (sleepers_ > 0) syscall(SYS_futex, &turn_, FUTEX_WAKE_PRIVATE, INT_MAX, nullptr, nullptr, 0);
    }

    template <typename There>
    void wait(There there)
    {
        for (const auto until = std::chrono::steady_clock::now() + std::chrono::microseconds(200); std::chrono::steady_clock::now() < until; std::this_thread::yield())
            if (there()) return;
        ++sleepers_;
        for (uint32_t turn; turn = turn_, !there();) syscall(SYS_futex, &turn_, FUTEX_WAIT_PRIVATE, turn, nullptr, nullptr, 0);
        --sleepers_;
    }

private:
    std::atomic<uint32_t> turn_{0};
    std::atomic<int> sleepers_{0};
    static_assert(sizeof(std::atomic<uint32_t>) == 4, "a futex is a word");
};

}  // namespace celty
