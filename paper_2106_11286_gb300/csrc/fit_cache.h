// What the driver answers about a kernel's occupancy at a launch shape on a
// device, kept for the life of the process: the questions cost a lattice's
// creation some 80 us, a fifth of it, and their answers depend on nothing else.
// One entry per variant and shape; any thread.
#pragma once

#include <cuda_runtime.h>

#include <map>
#include <mutex>
#include <tuple>

namespace hs {

template <typename F>
int cached_fit(const void *kernel, int ctas, int threads, F ask) {
    static std::mutex mu;
    static std::map<std::tuple<int, const void *, int, int>, int> known;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    const std::tuple<int, const void *, int, int> key{dev, kernel, ctas, threads};
    {
        std::lock_guard<std::mutex> lk(mu);
        const auto it = known.find(key);
        if (it != known.end()) return it->second;
    }
    const int v = ask();
    std::lock_guard<std::mutex> lk(mu);
    if (known.size() >= 4096) known.clear();  // bounded: shapes of a program that makes very many lattices
    known[key] = v;
    return v;
}

}  // namespace hs
