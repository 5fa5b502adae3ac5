"""The solve server's host-memory code (csrc/host_pool.h), compiled alone."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1710_02065_gb300", "csrc")


def run(tmp_path, program):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(program)
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr


COPY = r"""
#include <cstdio>
#include <new>
#include <system_error>
#include <vector>
#include "host_pool.h"
static int allowed;      // threads that can still be started
static bool no_memory;   // what the next one throws
struct Thread {
    std::thread t;
    Thread() = default;
    template <class F> explicit Thread(F f)
    {
        if (allowed == 0) {
            if (no_memory) throw std::bad_alloc();
            throw std::system_error(std::make_error_code(std::errc::resource_unavailable_try_again));
        }
        --allowed;
        t = std::thread(f);
    }
    Thread &operator=(Thread &&o) { t = std::move(o.t); return *this; }
    void join() { t.join(); }
};
int main()
{
    for (size_t n : {size_t(0), size_t(1), (size_t(1) << 19) - 1, size_t(1) << 19, (size_t(3) << 18) + 5, (size_t(1) << 21) + 3})
        for (int threads = 0; threads < 4; ++threads)
            for (int mem = 0; mem < 2; ++mem) {
                std::vector<double> a(n), b(n + 2, -1.0);
                for (size_t k = 0; k < n; ++k) a[k] = 0.5 * k;
                allowed = threads;
                no_memory = mem;
                rr::copy_host<Thread>(b.data() + 1, a.data(), n);
                if (b[0] != -1.0 || b[n + 1] != -1.0) return printf("wrote outside, n = %zu\n", n), 1;
                for (size_t k = 0; k < n; ++k)
                    if (b[k + 1] != a[k]) return printf("n = %zu, threads %d: element %zu\n", n, threads, k), 1;
            }
    return 0;
}
"""


def test_copy_with_any_number_of_threads_to_be_had(tmp_path):
    """Sizes around the thread count's steps; thread 0 to 3 fails to start, with
    either exception."""
    run(tmp_path, COPY)


POOL = r"""
#include <cstdio>
#include <cstdlib>
#include "host_pool.h"
static int allocs, frees;
static bool fail;
struct Fake {
    static double *alloc(size_t n) { return fail ? nullptr : (++allocs, (double *)malloc(n)); }
    static void free(double *b) { ++frees; ::free(b); }
};
#define CHECK(c) do { if (!(c)) { printf("line %d: %s (%d allocated, %d freed)\\n", __LINE__, #c, allocs, frees); return 1; } } while (0)
int main()
{
    {
        rr::HostBlocks<Fake> p(1000);
        double *a = p.take(300), *b = p.take(400), *c = p.take(500);
        CHECK(allocs == 3 && p.lent_bytes() == 1200 && p.kept_bytes() == 0);
        p.give(a);
        p.give(b);
        CHECK(frees == 0 && p.kept_bytes() == 700 && p.lent_bytes() == 500);
        p.give(c);  // displaces the first that came back
        CHECK(frees == 1 && p.kept_bytes() == 900);
        // a smaller request takes the smallest block of up to twice its size
        double *d = p.take(250);
        CHECK(d == b && allocs == 3 && p.lent_bytes() == 400 && p.kept_bytes() == 500);
        double *e = p.take(200);  // 500 > 2 x 200: a new one
        CHECK(e != c && allocs == 4);
        p.give(d);
        p.give(e);
        CHECK(frees == 2 && p.kept_bytes() == 600);
        // after the pool was filled with one size, requests of another find theirs kept
        double *big[4];
        for (double *&x : big) x = p.take(250);
        for (double *x : big) p.give(x);
        const int before = allocs;
        for (int k = 0; k < 10; ++k) {
            double *s[3] = {p.take(60), p.take(60), p.take(60)};
            for (double *x : s) p.give(x);
        }
        CHECK(allocs == before + 3);
        double *huge = p.take(1001);  // larger than all that is kept: not kept, nothing displaced
        const size_t kept = p.kept_bytes();
        p.give(huge);
        CHECK(p.kept_bytes() == kept && p.lent_bytes() == 0);
        fail = true;
        CHECK(p.take(5000) == nullptr && p.lent_bytes() == 0);
        fail = false;
        p.give(nullptr);
        p.set_keep(100);
        CHECK(p.kept_bytes() <= 100);
        p.set_keep(0);
        p.give(p.take(10));
        CHECK(p.kept_bytes() == 0 && allocs == frees);
        p.set_keep(1000);
        p.give(p.take(10));
    }
    CHECK(allocs == frees);
    return 0;
}
"""


def test_blocks_follow_the_sizes_in_use(tmp_path):
    """Reuse by smaller requests, displacement of the blocks that came back
    longest ago, failed allocations, changes of the bound; every block freed."""
    run(tmp_path, POOL)
