// Answers of a host query, remembered per device, kernel and launch shape in
// a fixed table: no memory is allocated and nothing is thrown, so that entry
// points which promise either may use it.  (No CUDA here.)
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <atomic>

namespace msc {

// Slots are claimed once and never change; a full table only means that the
// query is made again.  Several threads may ask at once.
class Remembered {
   public:
    // The answer of query(int* out) for the key: 0 when the query returned 0.
    template <typename Query>
    int get(int* out, int device, const void* kernel, int threads, size_t smem, Query query) {
        const size_t h0 = hash(device, kernel, threads, smem);
        for (size_t i = 0; i < kSlots; ++i) {
            Slot& s = slots_[(h0 + i) % kSlots];
            const int state = s.state.load(std::memory_order_acquire);
            if (state == kEmpty) break;
            if (state == kReady && s.device == device && s.kernel == kernel && s.threads == threads && s.smem == smem) {
                *out = s.answer;
                return 0;
            }
        }
        const int e = query(out);
        if (e != 0) return e;
        for (size_t i = 0; i < kSlots; ++i) {  // two threads may store one key twice: both hold its answer
            Slot& s = slots_[(h0 + i) % kSlots];
            int expect = kEmpty;
            if (!s.state.compare_exchange_strong(expect, kClaimed, std::memory_order_relaxed)) continue;
            s.device = device;
            s.kernel = kernel;
            s.threads = threads;
            s.smem = smem;
            s.answer = *out;
            s.state.store(kReady, std::memory_order_release);
            break;
        }
        return 0;
    }

   private:
    enum { kEmpty, kClaimed, kReady };
    struct Slot {
        std::atomic<int> state{kEmpty};
        int device = 0, threads = 0, answer = 0;
        const void* kernel = nullptr;
        size_t smem = 0;
    };
    static constexpr size_t kSlots = 1024;  // some 40 kernels and launch shapes per device
    Slot slots_[kSlots];

    static size_t hash(int device, const void* kernel, int threads, size_t smem) {
        uint64_t h = (uint64_t)(uintptr_t)kernel * 0x9e3779b97f4a7c15ull;
        h ^= (uint64_t)smem * 0xff51afd7ed558ccdull + (uint64_t)threads * 31u + (uint64_t)device;
        return (size_t)((h ^ (h >> 32)) % kSlots);
    }
};

}  // namespace msc
