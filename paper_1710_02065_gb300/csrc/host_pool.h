// host_pool.h -- host memory of the solve server's requests: copies between host
// buffers and the blocks kept for reuse.  Plain C++, no CUDA.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstring>
#include <map>
#include <thread>
#include <utility>
#include <vector>

namespace rr {

// Blocks of host memory lent to requests and kept for the next ones: allocating
// and freeing one per request costs more than its copies.  A request takes the
// smallest kept block of one to two times its size, or a new one.  At most
// `keep` bytes are kept: a block that comes back displaces those that came back
// longest ago, so the kept ones follow the sizes in use.  Alloc: static
// double *alloc(size_t bytes) (null: no memory) and void free(double *).
template <class Alloc>
class HostBlocks {
public:
    explicit HostBlocks(size_t keep) : keep_(keep) {}
    HostBlocks(const HostBlocks &) = delete;
    HostBlocks &operator=(const HostBlocks &) = delete;
    ~HostBlocks() { set_keep(0); }  // (lent blocks have been given back)

    // A block of at least `bytes` (null: no memory)
    double *take(size_t bytes)
    {
        auto best = kept_.end();
        for (auto it = kept_.begin(); it != kept_.end(); ++it)
            if (it->second >= bytes && it->second <= 2 * bytes && (best == kept_.end() || it->second < best->second))
                best = it;
        const bool reuse = best != kept_.end();
        const std::pair<double *, size_t> b = reuse ? *best : std::make_pair(Alloc::alloc(bytes), bytes);
        if (!b.first) return nullptr;
        try {
            lent_.insert(b);
        } catch (...) {
            if (!reuse) Alloc::free(b.first);
            return nullptr;
        }
        if (reuse) {
            kept_.erase(best);
            kept_bytes_ -= b.second;
        }
        lent_bytes_ += b.second;
        return b.first;
    }

    // Give a block back (null: none)
    void give(double *b)
    {
        const auto it = lent_.find(b);
        if (it == lent_.end()) return;
        const size_t size = it->second;
        lent_.erase(it);
        lent_bytes_ -= size;
        if (size <= keep_) {
            drop_to(keep_ - size);
            try {
                kept_.emplace_back(b, size);
                kept_bytes_ += size;
                return;
            } catch (...) {
            }
        }
        Alloc::free(b);
    }

    void set_keep(size_t keep)
    {
        keep_ = keep;
        drop_to(keep);
    }
    size_t lent_bytes() const { return lent_bytes_; }
    size_t kept_bytes() const { return kept_bytes_; }

private:
    void drop_to(size_t bytes)
    {
        auto it = kept_.begin();
        for (; it != kept_.end() && kept_bytes_ > bytes; ++it) {
            Alloc::free(it->first);
            kept_bytes_ -= it->second;
        }
        kept_.erase(kept_.begin(), it);
    }

    std::vector<std::pair<double *, size_t>> kept_;  // in the order in which they came back
    std::map<double *, size_t> lent_;
    size_t kept_bytes_ = 0, lent_bytes_ = 0, keep_;
};

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
