// What a kernel needs once on each device before it is launched, whichever
// thread comes first: the opt-in to its dynamic shared memory, and how many of
// its CTAs an SM holds.  The attribute belongs to the kernel on the current
// device, and a smaller value set later would take a larger one away from a
// launch of another thread, so it only grows, under a lock (taken once per
// launch, 20 ns).  Nothing of CUDA is named here: callers pass what sets it.
#pragma once

#include <cstddef>
#include <map>
#include <mutex>
#include <utility>

namespace sivf {

struct KernelSetup {
    // set(bytes) -> whether it took, called with more than the device has
    template <class Set>
    void opt_in(int device, size_t smem, size_t builtin, Set set)
    {
        std::lock_guard<std::mutex> g(m);
        size_t &have = smem_of.try_emplace(device, builtin).first->second;
        if (smem > have && set(smem)) have = smem;
    }
    // count() -> CTAs per SM at this much shared memory
    template <class Count>
    int resident(int device, size_t smem, Count count)
    {
        std::lock_guard<std::mutex> g(m);
        auto it = ctas_of.find({device, smem});
        if (it == ctas_of.end()) it = ctas_of.emplace(std::make_pair(device, smem), count()).first;
        return it->second;
    }

private:
    std::mutex m;
    std::map<int, size_t> smem_of;
    std::map<std::pair<int, size_t>, int> ctas_of;
};

}  // namespace sivf
