// hfs_resident.h -- what a launch site remembers of its kernel's occupancy.
#pragma once

#include <stdint.h>

#include <atomic>

namespace hfs {

// CTAs of a persistent grid, by device, threads of a CTA and its shared memory: the
// last eight of a launch site.  Models of different sizes share a kernel, and the
// same shared memory goes with several CTA sizes (the projection stage at 16 channels
// and 16 modes: 32 points with proj 128 and 64 points with proj 64, 10944 bytes), so
// both are part of the key; with one entry and no thread count the second such model
// ran on the first one's grid, and others in turn asked at every launch.  An entry is
// one word, so threads need no lock: a race only asks twice.
class ResidentSlot {
public:
    // ctas of the key, from ask(int *ctas) (0: success) where it is not remembered
    template <typename Ask> int get(int dev, int threads, uint64_t smem, Ask ask, int *ctas)
    {
        const bool keep = dev >= 0 && dev < 64 && threads > 0 && threads <= 1024 && smem < (1u << 18);
        const uint64_t key = (uint64_t)1 << 63 | (uint64_t)dev << 48 | (uint64_t)threads << 36 | smem << 18;
        if (keep)
            for (auto &e : entry_) {
                const uint64_t v = e.load(std::memory_order_relaxed);
                if ((v & ~kCtas) == key) {
                    *ctas = (int)(v & kCtas);
                    return 0;
                }
            }
        const int status = ask(ctas);
        if (status == 0 && keep && *ctas >= 0 && (uint64_t)*ctas <= kCtas)
            entry_[next_.fetch_add(1, std::memory_order_relaxed) % kEntries].store(key | (uint64_t)*ctas, std::memory_order_relaxed);
        return status;
    }

private:
    static constexpr uint64_t kCtas = (1u << 18) - 1;
    static constexpr unsigned kEntries = 8;
    std::atomic<uint64_t> entry_[kEntries] = {};
    std::atomic<unsigned> next_{0};
};

}  // namespace hfs
