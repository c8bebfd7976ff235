// serve_result.h -- what a serving launch publishes to the host for a slot, and
// how the host reads it.  Plain C++: the tests run it against a host thread.
#pragma once

namespace proxmf {

struct ServeResult {         // host-mapped
    int done;                // 1 once retired
    int iters;
    double F;                // F of the state before the last step
};

enum class ServeSlotState { running, finished, timed_out };

// State of a slot in flight.  `status` is the word that a launch sets when one of
// its waits runs out; its tiles are then unwritten, and the launch that ends the
// iteration may still set `done` from what was there before.  The device writes
// status before done, so the host reads done first: a finished slot is one that
// was done with the word still clear.  The load of done acquires: the status word,
// iters and F are read after it on a host that reorders loads (Arm) too.
inline ServeSlotState serve_slot_state(const ServeResult &r, const volatile int *status) {
    if (__atomic_load_n(&r.done, __ATOMIC_ACQUIRE) == 0) return ServeSlotState::running;
    return __atomic_load_n(status, __ATOMIC_RELAXED) != 0 ? ServeSlotState::timed_out : ServeSlotState::finished;
}

}  // namespace proxmf
