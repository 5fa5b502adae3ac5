// host_pool.h -- host memory of the solve server's requests: copies between host
// buffers and the blocks kept for reuse.  Plain C++, no CUDA.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstring>
#include <thread>

namespace rr {

// Copy n doubles; large copies by up to four threads (one core's copy rate is a
// fraction of the memory's).  Does not throw: the parts for which there is no
// thread to be had are copied here.
template <class Thread = std::thread>
void copy_host(double *dst, const double *src, size_t n)
{
    constexpr size_t kPart = size_t(1) << 18;  // doubles a thread is worth starting for
    constexpr size_t kThreads = 4;
    const size_t parts = std::max<size_t>(1, std::min(kThreads, n / kPart));
    auto copy = [=](size_t a, size_t b) {
        if (b > a) std::memcpy(dst + a, src + a, (b - a) * sizeof(double));
    };
    Thread th[kThreads - 1];
    size_t started = 0;
    try {
        for (; started + 1 < parts; ++started) {
            const size_t k = started + 1, a = n * k / parts, b = n * (k + 1) / parts;
            th[started] = Thread([=] { copy(a, b); });
        }
    } catch (...) {
    }
    copy(0, n / parts);
    copy(n * (started + 1) / parts, n);
    for (size_t k = 0; k < started; ++k) th[k].join();
}

}  // namespace rr
