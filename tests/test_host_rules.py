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


PLANS = """
#include "plan.h"
struct Held { int c2, c4, c8; int operator()(int ctas) const { return ctas == 2 ? c2 : (ctas == 4 ? c4 : c8); } };
// -> CTAs per cluster, 0: two launches
extern "C" int fused(long M, long N, long K, int block, int bits, int mult, int sms, int c2, int c4, int c8) {
    const fq::FusedPlan f = fq::plan_fused(M, N, K, block, bits, mult != 0, sms, Held{c2, c4, c8});
    return f.lanes ? 1 << f.ctas_shift : 0;
}
// -> 100 * tokens per cluster + CTAs per cluster, 0: two launches
extern "C" int composite(long M, long K, int elem, int beta, int sms, int c2, int c4, int c8) {
    const fq::CompositePlan f = fq::plan_composite(M, K, elem, beta, sms, Held{c2, c4, c8});
    return f.tok ? 100 * f.tok + (1 << f.ctas_shift) : 0;
}
"""
B200 = (148, 74, 36, 14)       # multiprocessors, clusters of 2, 4 and 8 CTAs that a whole device holds


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    return compile_host(tmp_path_factory.mktemp("plans"), "plans", PLANS)


def test_one_launch_paths_need_clusters_that_can_be_placed(plans):
    def fused(M, N, K, block, bits, device=B200):
        return plans.fused(M, N, K, block, bits, 0, *device)

    assert fused(50, 1024, 1024, 64, 4) == 8 and fused(20, 1024, 1024, 64, 8) == 4 and fused(20, 1024, 512, 64, 8) == 2
    assert fused(8, 64, 256, 64, 4) == 1
    part = (16, 8, 0, 0)       # a part of a device: pairs only
    assert fused(50, 128, 1024, 64, 4, part) == 0 and fused(20, 128, 1024, 64, 8, part) == 0
    assert fused(20, 128, 512, 64, 8, part) == 2 and fused(8, 64, 256, 64, 4, (16, 0, 0, 0)) == 1

    def composite(M, K, elem, beta, device=B200):
        return plans.composite(M, K, elem, beta, *device)

    assert composite(816, 2048, 2, 64) == 1602 and composite(576, 2048, 2, 64) == 1604 and composite(16, 2048, 2, 64) == 1608
    assert composite(20, 4096, 4, 128) == 808                                    # binary32 rows: eight tokens, eight CTAs
    for device in (part, (16, 0, 0, 0)):
        for M, K, elem, beta in [(816, 2048, 2, 64), (16, 2048, 2, 64), (20, 4096, 4, 128), (17, 512, 4, 16), (9, 8192, 4, 64)]:
            tok, ctas = divmod(composite(M, K, elem, beta, device), 100)
            assert ctas <= (2 if device[1] else 1), (M, K, elem, beta, device)
    assert composite(20, 4096, 4, 128, (16, 0, 0, 0)) == 0                       # fits in clusters only: two launches
