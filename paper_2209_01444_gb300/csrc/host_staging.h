// The process's page-locked staging buffer for transfers to and from pageable
// host memory (defined in lbm_api.cu): at most 2 x kPinHalf bytes, allocated on
// first use, kept until exit; a call holds the mutex while it uses it.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <mutex>
#include <thread>
#include <vector>

namespace lbm {

constexpr size_t kPinHalf = (size_t)32 << 20;

struct PinnedStaging {
    std::mutex mu;
    float* p = nullptr;
    size_t bytes = 0;
};
extern PinnedStaging g_pinned;

// The buffer grown to at least `bytes` (<= 2 kPinHalf); the caller holds
// g_pinned.mu.  Null, with the error in *e, when page-locked memory cannot be had.
float* pinned_staging(size_t bytes, cudaError_t* e);

// Runs fn(i0, i1) over the range [0, n) on up to 16 host threads, at least
// `least` indices each.
template <class Fn>
void parallel_range(long long n, long long least, Fn fn)
{
    static const long long most = std::min(std::thread::hardware_concurrency(), 16u);  // (a read of /sys each time)
    const int nt = (int)std::max<long long>(1, std::min(most, n / std::max(1LL, least)));
    if (nt == 1) {
        fn(0LL, n);
        return;
    }
    std::vector<std::thread> pool;
    int started = 0;
    try {
        pool.reserve(nt);
        for (; started < nt - 1; ++started) pool.emplace_back(fn, n * started / nt, n * (started + 1) / nt);
    } catch (...) {  // no more threads: the rest runs here
    }
    fn(n * started / nt, n);
    for (std::thread& th : pool) th.join();
}

}  // namespace lbm
