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
