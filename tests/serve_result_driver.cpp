// A host thread publishes slots as the device does (status word, then iters and
// F, then done); the reader must never take a slot whose status word was set for
// finished, and must see the iters and F of those that are.
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>

#include "serve_result.h"

using namespace proxmf;

int main(int argc, char **) {
    const int n = argc > 1 ? 20000 : 400000;
    std::atomic<int> at{-1};   // the slot the reader polls: published while it does
    std::vector<ServeResult> res(n, ServeResult{0, 0, 0.0});
    std::vector<int> status(n, 0);
    std::thread device([&] {
        for (int i = 0; i < n; ++i) {
            while (at.load(std::memory_order_relaxed) < i) {}
            for (volatile int d = 0; d < i % 37; ++d) {}
            if (i % 2) __atomic_store_n(&status[i], -5, __ATOMIC_RELAXED);
            res[i].iters = i;
            res[i].F = 0.5 * i;
            __atomic_store_n(&res[i].done, 1, __ATOMIC_RELEASE);
        }
    });
    long bad = 0;
    for (int i = 0; i < n; ++i) {
        at.store(i, std::memory_order_relaxed);
        ServeSlotState s;
        do s = serve_slot_state(res[i], &status[i]);
        while (s == ServeSlotState::running);
        if (s != (i % 2 ? ServeSlotState::timed_out : ServeSlotState::finished)) ++bad;
        if (s == ServeSlotState::finished && (res[i].iters != i || res[i].F != 0.5 * i)) ++bad;
    }
    device.join();
    if (bad) std::printf("%ld of %d slots read wrongly\n", bad, n);
    return bad ? 1 : 0;
}
