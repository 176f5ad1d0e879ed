// gs_occupancy.h -- the answers of occupancy queries, kept.  Plain C++: host code only.
#pragma once

#include <cstddef>
#include <mutex>

namespace gs {

// How many CTAs of a kernel a device holds at once, by kernel, CTA size, dynamic
// shared memory and device: a plan's launches of one kernel alternate between
// sizes, and threads may launch on several devices.  ask() is called once per key
// (again while the table is full); answers below 1 are not kept.
class OccupancyCache {
public:
    template <class Ask>
    int get(const void* kernel, int threads, size_t smem, int dev, Ask ask) {
        std::lock_guard<std::mutex> lock(mu_);
        for (int i = 0; i < used_; ++i) {
            const Entry& e = entries_[i];
            if (e.kernel == kernel && e.smem == smem && e.threads == threads && e.dev == dev)
                return e.ctas;
        }
        const int ctas = ask();
        if (ctas >= 1 && used_ < kEntries) entries_[used_++] = {kernel, smem, threads, dev, ctas};
        return ctas;
    }

private:
    static constexpr int kEntries = 256;
    struct Entry {
        const void* kernel;
        size_t smem;
        int threads, dev, ctas;
    };
    Entry entries_[kEntries] = {};
    int used_ = 0;
    std::mutex mu_;
};

}  // namespace gs
