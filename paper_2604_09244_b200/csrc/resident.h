// How many clusters of a kernel run at once, remembered per device.
//
// The runtime's occupancy calculator takes longer than a launch, and its answer depends on the kernel, the cluster size,
// the block size, the shared memory and the device: devices of one machine may differ in multiprocessors and in how these are grouped.
// One object per kernel; host threads may share it (an entry holds question and answer in one word).
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <atomic>

namespace mvla {

class ResidentClusters {
public:
    static constexpr int kDevices = 64, kSizes = 16, kMaxThreads = 1024, kMaxCount = 0xFFFF;
    // The answer kept for this question, or 0.
    int find(int device, int cluster, size_t smem, int threads = 0) const
    {
        if (!covers(device, cluster, threads)) return 0;
        const uint64_t e = last_[device][cluster][way(threads)].load(std::memory_order_relaxed);
        return e >> 16 == question(threads, smem) ? static_cast<int>(e & kMaxCount) : 0;
    }
    void keep(int device, int cluster, size_t smem, int count, int threads = 0)
    {
        if (covers(device, cluster, threads) && count > 0 && count <= kMaxCount)
            last_[device][cluster][way(threads)].store(question(threads, smem) << 16 | static_cast<uint32_t>(count), std::memory_order_relaxed);
    }

private:
    static bool covers(int device, int cluster, int threads)
    {
        return device >= 0 && device < kDevices && cluster >= 0 && cluster < kSizes && threads >= 0 && threads <= kMaxThreads;
    }
    static uint64_t question(int threads, size_t smem) { return static_cast<uint64_t>(smem + 1) << 16 | static_cast<uint32_t>(threads); }
    // (a kernel that is launched with two block sizes in turn, two warps apart, keeps an answer for each)
    static int way(int threads) { return threads / 64 % 2; }
    // (shared memory + 1, threads, answer) of the last question with this cluster size: a program's calls alternate between few
    std::atomic<uint64_t> last_[kDevices][kSizes][2] = {};
};

}  // namespace mvla
