// status_words.cuh -- who holds which of the device status words that entry points without a context share.
//
// A kernel whose bounded wait gives up sets a bit in its call's word.  With one word for all calls, a call
// on another thread or stream would clear it, or take it for its own; so each call holds a word of its own
// until its work is complete.  (Host code only.)
#pragma once

#include <atomic>
#include <thread>

namespace soap {

template <int N>
class StatusWords {
public:
    // The index of a word that no other call holds; waits while all are held (a holder's kernels end).
    int claim() {
        while (true) {
            for (int i = 0; i < N; i++)
                if (!held_[i].exchange(true, std::memory_order_acquire)) return i;
            std::this_thread::yield();
        }
    }
    void give_back(int i) { held_[i].store(false, std::memory_order_release); }

private:
    std::atomic<bool> held_[N] = {};
};

}  // namespace soap
