// How many clusters of a kernel run at once, remembered per device.
//
// The runtime's occupancy calculator takes longer than a launch, and its answer depends on the kernel, the cluster size,
// the shared memory and the device: devices of one machine may differ in multiprocessors and in how these are grouped.
// One object per kernel; host threads may share it (an entry holds question and answer in one word).
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <atomic>

namespace mvla {

class ResidentClusters {
public:
    static constexpr int kDevices = 64, kSizes = 16;
    // The answer kept for this question, or 0.
    int find(int device, int cluster, size_t smem) const
    {
        if (!covers(device, cluster)) return 0;
        const uint64_t e = last_[device][cluster].load(std::memory_order_relaxed);
        return (e >> 32) == smem + 1 ? static_cast<int>(e & 0xFFFFFFFFu) : 0;
    }
    void keep(int device, int cluster, size_t smem, int count)
    {
        if (covers(device, cluster) && count > 0)
            last_[device][cluster].store((static_cast<uint64_t>(smem + 1) << 32) | static_cast<uint32_t>(count), std::memory_order_relaxed);
    }

private:
    static bool covers(int device, int cluster) { return device >= 0 && device < kDevices && cluster >= 0 && cluster < kSizes; }
    // (shared memory + 1, answer) of the last question with this cluster size: a program's calls alternate between few
    std::atomic<uint64_t> last_[kDevices][kSizes] = {};
};

}  // namespace mvla
