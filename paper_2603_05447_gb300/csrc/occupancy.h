// occupancy.h -- what a launch needs to know of a kernel, asked once: whether it
// may have more than 48 KB of dynamic shared memory, and how many of its blocks
// an SM holds.  Both belong to a device, and a process may have grids on
// several, so they are kept per device and kernel.  Host code only.
#pragma once

#include <cstddef>
#include <map>
#include <mutex>
#include <unordered_map>
#include <utility>

namespace gpe {

class Occupancy {
  public:
    // Resident blocks an SM of `kernel` on `device` with smem bytes of dynamic
    // shared memory.  prepare() lets the kernel have its shared memory and says
    // whether that worked; query() gives the blocks (below 1: failed).  What
    // failed is tried again at the next call; the answer is then 1, and the
    // launch itself reports what is wrong.
    template <typename PREPARE, typename QUERY>
    int blocks(int device, const void *kernel, size_t smem, PREPARE prepare, QUERY query)
    {
        std::lock_guard<std::mutex> lk(mu_);
        Kernel &k = known_[{device, kernel}];
        if (!k.prepared) k.prepared = prepare();
        const auto it = k.per_sm.find(smem);
        if (it != k.per_sm.end()) return it->second;
        const int per = query();
        if (per < 1) return 1;
        if (k.prepared && k.per_sm.size() < MAX_SIZES) k.per_sm[smem] = per;
        return per;
    }

  private:
    static constexpr size_t MAX_SIZES = 256;  // shared-memory sizes remembered of a kernel
    struct Kernel {
        bool prepared = false;
        std::unordered_map<size_t, int> per_sm;
    };
    std::mutex mu_;
    std::map<std::pair<int, const void *>, Kernel> known_;
};

}  // namespace gpe
