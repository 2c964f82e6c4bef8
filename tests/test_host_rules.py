"""Host-side rules of the library, compiled by themselves with g++ and called without a device."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_24433_b200", "csrc")


def compile_host(folder, name, source):
    src, lib = os.path.join(str(folder), name + ".cpp"), os.path.join(str(folder), name + ".so")
    with open(src, "w") as f:
        f.write(source)
    subprocess.run(["g++", "-std=c++17", "-O2", "-Wall", "-Werror", "-fPIC", "-shared", "-pthread", "-I", CSRC, src, "-o", lib], check=True)
    return ctypes.CDLL(lib)


OPT_IN = """
#include "smem_opt_in.h"
#include <atomic>
#include <chrono>
#include <thread>
#include <vector>
// `threads` host threads launch one kernel with as many sizes; -> launches that found the attribute below their size
extern "C" int races(int threads, int refuse) {
    fq::SmemOptIn table;
    std::atomic<size_t> attribute{0};
    std::atomic<int> ready{0}, bad{0};
    auto one = [&](int i) {
        const size_t bytes = 1000 * (size_t)(1 + (i * 7) % threads);
        ++ready;
        while (ready < threads) {}
        auto set = [&](size_t n) {
            std::this_thread::sleep_for(std::chrono::microseconds(200 + 37 * ((i * 5) % threads)));
            if (refuse && n > (size_t)refuse) return 1;
            attribute = n;
            std::this_thread::sleep_for(std::chrono::microseconds(37 * i));
            return 0;
        };
        for (int k = 0; k < 3; ++k) {
            const int e = table.raise(&table, bytes, set);
            if (e == 0 ? attribute < bytes : !(refuse && bytes > (size_t)refuse)) ++bad;
        }
    };
    std::vector<std::thread> pool;
    for (int i = 0; i < threads; ++i) pool.emplace_back(one, i);
    for (auto& t : pool) t.join();
    return bad;
}
"""


@pytest.mark.parametrize("threads,refuse", [(2, 0), (8, 0), (8, 4500)])
def test_shared_memory_opt_in_from_several_threads(tmp_path, threads, refuse):
    """A thread that was told "success" finds the attribute at its size or above; a refused size is not recorded."""
    lib = compile_host(tmp_path, "opt_in", OPT_IN)
    assert sum(lib.races(threads, refuse) for _ in range(20)) == 0
