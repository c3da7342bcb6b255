// cluster_fit.h -- whether a thread-block cluster of a given shape can run here.
//
// A cluster's CTAs have to be resident at once, next to each other: the sizes
// above 8 CTAs need not be available (a partition of the device, SMs taken out),
// and a launch that cannot be had is an error.  The question is asked once per
// device, kernel and shape; without a place the step kernels and the four
// kernels of the list build are launched, which give the same bits.
#pragma once

#include <cstddef>
#include <map>
#include <mutex>
#include <tuple>

namespace gld {

constexpr int kClThreads = 512;  // threads of a CTA
constexpr int kClMaxCtas = 16;   // non-portable above 8

// CTAs that give each of n particles `lanes` threads, a power of two up to 16.
inline int cluster_ctas(int n, int lanes)
{
    int c = 1;
    while (c < kClMaxCtas && c * (kClThreads / lanes) < n) c *= 2;
    return c;
}

// Lanes per particle of a cluster of `ctas` CTAs that steps n particles.
inline int cluster_lanes(int n, int ctas)
{
    return ctas * kClThreads / 8 >= n ? 8 : ctas * kClThreads / 4 >= n ? 4 : 2;
}

// Totals of the cell scan: one per chunk of 512 cells, or one per CTA of the list
// build in a cluster, whichever is more.
inline int scan_totals(int ncells)
{
    const int chunks = (ncells + 511) / 512;
    return chunks > kClMaxCtas ? chunks : kClMaxCtas;
}

class ClusterFit {
public:
    // ask(smem): clusters that can be resident at once (0: none, or it failed).
    // Shared memory counts in steps of 4 KB, so few answers are kept.
    template <class Ask>
    bool operator()(int dev, const void* kern, int ctas, size_t smem, Ask&& ask)
    {
        const size_t asked = (smem + 4095) / 4096 * 4096;
        std::lock_guard<std::mutex> lock(mu);
        const auto key = std::make_tuple(dev, kern, ctas, asked);
        auto it = known.find(key);
        if (it == known.end()) it = known.emplace(key, ask(asked) > 0).first;
        return it->second;
    }

private:
    std::mutex mu;
    std::map<std::tuple<int, const void*, int, size_t>, bool> known;
};

}  // namespace gld
