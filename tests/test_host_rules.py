"""Host-side rules of the library, compiled by themselves with g++ and called without a device."""
import ctypes
import os
import subprocess

import pytest

import test_gpu_edges as edges
import test_gpu_parity as parity

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
// -> 100 * rounds + CTAs per cluster, 0: two launches
extern "C" int fused(long M, long N, long K, int block, int bits, int mult, int sms, int c2, int c4, int c8, int* grid) {
    const fq::FusedPlan f = fq::plan_fused(M, N, K, block, bits, mult != 0, sms, Held{c2, c4, c8});
    *grid = f.grid;
    return f.lanes ? 100 * f.rounds + (1 << f.ctas_shift) : 0;
}
// -> 100 * tokens per cluster + CTAs per cluster, 0: two launches
extern "C" int composite(long M, long K, int elem, int beta, int sms, int c2, int c4, int c8, int* grid) {
    const fq::CompositePlan f = fq::plan_composite(M, K, elem, beta, sms, Held{c2, c4, c8});
    *grid = (int)f.grid;
    return f.tok ? 100 * f.tok + (1 << f.ctas_shift) : 0;
}
// -> channels per thread of the streamed prologue, 0: the register kernel
extern "C" int ring(long M, long K, int elem, int gated, int bytes_out, int mult, int after, int block, int sms) {
    return fq::plan_ring(M, K, elem, gated, bytes_out, mult, after, block, sms).e;
}
// scratch < 0: as much as the plan without clusters asks for
extern "C" void gemm(long M, long N, long K, int bits, long scratch, int sms, int c2, int c4, int c8, int* out) {
    const Held held{c2, c4, c8};
    const size_t asks = fq::plan_gemm(M, N, K, bits, sms, (size_t)-1, false, held).scratch;
    const fq::GemmPlan f = fq::plan_call(M, N, K, bits, sms, scratch < 0 ? asks : (size_t)scratch, held);
    const fq::GemmRings r = fq::gemm_rings(f, bits, K);
    const int v[] = {fq::plan_stream(M, N, K, bits, sms, held), f.bt, f.ctas, f.split, f.cluster, f.scratch > 0, r.fits, r.atoms, r.stages,
                     r.stages_p, r.stages_w, r.slot_first, (int)r.smem, r.tmem_cols, f.stack, f.epi};
    for (int i = 0; i < 16; ++i) out[i] = v[i];
}
"""
B200 = (148, 74, 36, 14)       # multiprocessors, clusters of 2, 4 and 8 CTAs that one whole device holds
WHOLE = [B200, (148, 74, 33, 15)]                        # ... and another, whose SMs are grouped otherwise
GEMM = "stream bt ctas split cluster scratch fits atoms stages stages_p stages_w slot_first smem tmem_cols stack epi".split()


class Plans:
    def __init__(self, lib, device=B200):
        self.lib, self.device, self.grid = lib, device, 0

    def on(self, device):
        return Plans(self.lib, device)

    def fused(self, M, K, N, block, bits, mult=False, device=None):
        grid = ctypes.c_int()
        r = self.lib.fused(ctypes.c_long(M), ctypes.c_long(N), ctypes.c_long(K), block, bits, int(mult), *(device or self.device), ctypes.byref(grid))
        self.grid = grid.value
        return r

    def composite(self, M, K, dtype, beta, device=None):
        grid = ctypes.c_int()
        r = self.lib.composite(ctypes.c_long(M), ctypes.c_long(K), 2 if dtype == "bf16" else 4, beta, *(device or self.device), ctypes.byref(grid))
        self.grid = grid.value
        return r

    def ring(self, M, K, dtype, block, bytes_out, form="plain", gated=False):
        return self.lib.ring(ctypes.c_long(M), ctypes.c_long(K), 2 if dtype == "bf16" else 4, int(gated), int(bytes_out),
                             int(form != "plain"), int(form == "after"), block, B200[0])

    def gemm(self, M, K, N, bits, scratch=-1, device=None):
        out = (ctypes.c_int * len(GEMM))()
        self.lib.gemm(ctypes.c_long(M), ctypes.c_long(N), ctypes.c_long(K), bits, ctypes.c_long(scratch), *(device or self.device), out)
        return dict(zip(GEMM, out))


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    return Plans(compile_host(tmp_path_factory.mktemp("plans"), "plans", PLANS))


def test_one_launch_paths_need_clusters_that_can_be_placed(plans):
    assert plans.fused(50, 1024, 1024, 64, 4) == 108 and plans.fused(20, 1024, 1024, 64, 8) == 104
    assert plans.fused(20, 512, 1024, 64, 8) == 102 and plans.fused(8, 256, 64, 64, 4) == 101
    part, none = (16, 8, 0, 0), (16, 0, 0, 0)          # parts of a device: pairs only, and no clusters at all
    assert plans.fused(50, 1024, 128, 64, 4, device=part) == 0 and plans.fused(20, 1024, 128, 64, 8, device=part) == 0
    assert plans.fused(20, 512, 128, 64, 8, device=part) == 102 and plans.fused(8, 256, 64, 64, 4, device=none) == 101

    assert plans.composite(816, 2048, "bf16", 64) == 1602 and plans.composite(16, 2048, "bf16", 64) == 1608
    assert plans.composite(20, 4096, "f32", 128) == 808
    for device in (part, none):
        for M, K, dtype, beta in [(816, 2048, "bf16", 64), (16, 2048, "bf16", 64), (20, 4096, "f32", 128), (17, 512, "f32", 16)]:
            assert plans.composite(M, K, dtype, beta, device) % 100 <= (2 if device[1] else 1), (M, K, dtype, beta, device)
    assert plans.composite(20, 4096, "f32", 128, none) == 0      # fits in clusters only: two launches
    for M, K, N, bits in edges.CLUSTER_SPLIT + edges.SCRATCH_SPLIT:
        p = plans.gemm(M, K, N, bits, scratch=0, device=none)
        assert p["fits"] and p["ctas"] == 1 and p["split"] == 1


@pytest.mark.parametrize("device", WHOLE)
def test_sizes_of_the_device_tests_take_the_routes_they_stand_for(plans, device):
    plans = plans.on(device)
    for M, K, N, block, bits, _, smooth, _ in edges.ONE_LAUNCH:
        assert plans.fused(M, K, N, block, bits, smooth), (M, K, N)
        assert plans.grid <= B200[0]
    assert [plans.fused(*c[:5]) for c in edges.ONE_LAUNCH if c[1] > 1700] == [208, 208, 208, 208]       # two rounds
    assert not plans.fused(8, 1024, 3080, 64, 4) and not plans.fused(32, 1024, 4104, 64, 4) and not plans.fused(33, 1024, 1032, 64, 4)
    assert not plans.fused(33, 512, 1544, 64, 8) and not plans.fused(33, 256, 128, 64, 4)
    assert not plans.fused(33, 2176, 128, 64, 4) and not plans.fused(32, 4224, 128, 64, 4) and not plans.fused(65, 1024, 128, 64, 4)
    for M, K, block, bits in edges.FEW_UNITS:
        ctas = plans.fused(M, K, 200, block, bits) % 100
        assert K // max(block, 128) < ctas, (M, K)
    for M, K, bits, call in edges.TO_AND_FRO[:3]:
        assert plans.fused(M, K, K, 64, bits)
    assert not plans.gemm(24, 4096, 4096, 4)["stream"] and not plans.fused(24, 4096, 4096, 64, 4) and plans.gemm(12, 4096, 4096, 8)["stream"]

    for M, K, N in edges.ODD_RINGS:
        p = plans.gemm(M, K, N, 4)
        assert p["fits"] and p["slot_first"] and p["stages_p"] % 2 == 1 and not p["stream"], (M, K, N, p)
    rings = [(p["stages_p"], p["stages_w"], p["split"]) for p in (plans.gemm(*c, 4) for c in edges.ODD_RINGS)]
    assert rings == [(3, 3, 1), (5, 5, 1), (5, 4, 1), (5, 4, 4)]
    for M, K, N, bits in edges.CLUSTER_SPLIT:
        p = plans.gemm(M, K, N, bits, scratch=0)
        assert p["fits"] and p["cluster"] and p["split"] > 1 and not p["stream"], (M, K, N, bits, p)
        assert plans.gemm(M, K, N, bits)["cluster"]
    for M, K, N, bits in edges.SCRATCH_SPLIT:
        p = plans.gemm(M, K, N, bits)
        assert p["fits"] and p["scratch"] and p["split"] > 1 and not p["cluster"] and not p["stream"], (M, K, N, bits, p)
        assert not plans.gemm(M, K, N, bits, scratch=0)["scratch"]
    assert plans.gemm(*edges.SCRATCH_SPLIT[-1])["ctas"] == 2
    for M, K, N, warps in edges.W8_EPILOGUE:
        p = plans.gemm(M, K, N, 8)
        assert p["fits"] and p["split"] == 1 and p["epi"] == warps and not p["stream"], (M, K, N, p)
    assert [plans.gemm(M, K, N, 8)["ctas"] for M, K, N, _ in edges.W8_EPILOGUE] == [1] * 5 + [2] * 6
    assert all(plans.gemm(*c)["epi"] == 8 for c in edges.CLUSTER_SPLIT + edges.SCRATCH_SPLIT)
    assert all(plans.gemm(*c, 4)["ctas"] == 2 for c in edges.W4_PAIRS) and all(plans.gemm(*c, 4)["ctas"] == 1 for c in edges.W4_SINGLE)

    for M, K, beta, _, dtype, _, lead in edges.COMPOSITE:
        assert (plans.composite(M, K, dtype, beta) == 0) == (K == 8192), (M, K, beta)
    assert plans.composite(700, 1024, "bf16", 32) and plans.grid > B200[0]
    assert plans.composite(16 * device[2], 2048, "bf16", 64) == 1604 and plans.grid == 4 * device[2]
    assert plans.composite(16 * device[2] + 1, 2048, "bf16", 64) == 1602
    assert [bool(plans.ring(M, K, "bf16", block, bits == 8, gated=True)) for M, K, block, bits, _ in edges.GATED] == [True, False, True]
    for M, K, block, bits, dtype, form in edges.PROLOGUE:
        e = plans.ring(M, K, dtype, block, bits == 8, form)
        assert bool(e) == (M != 1300) and all(plans.ring(40, K, dtype, block, b, form) == 0 for b in (False, True)), (M, K, e)
        assert plans.ring(M, K, dtype, block, True, form) == e                  # the one-call route writes a byte per code
        assert M == 1300 or plans.ring(M - 1, K, dtype, block, True, form) == 0
    # prologues that are shorter in a call of their own and longer in front of a GEMM stay in the register kernel
    assert not any(plans.ring(M, K, "bf16", 128, True, form) for M, K in ((700, 2048), (816, 2048), (1156, 2048), (320, 4096), (160, 8192))
                   for form in ("plain", "smooth"))
    assert plans.ring(1170, 10240, "bf16", 128, True, "smooth")


@pytest.mark.parametrize("device", WHOLE + [(16, 8, 0, 0)])
def test_rings_of_every_plan_fit(plans, device):
    """Shared and tensor memory within the SM's, a ring that the unpack sets cannot misread, and room left for no second CTA of
    the short-batch kernel (77 KB) beside a cluster."""
    for bits in (4, 8):
        for K in (32, 128, 160, 2048, 4096, 8192, 8256, 16384, 32768):
            for M in (1, 16, 17, 50, 64, 65, 112, 128, 129, 208, 256, 300, 816, 1000, 4096, 20000):
                for N in (8, 128, 136, 1024, 2048, 4104, 8192, 16384):
                    for scratch in (0, -1):
                        p = plans.gemm(M, K, N, bits, scratch, device)
                        assert p["fits"] and p["smem"] <= 227 * 1024 and p["tmem_cols"] <= 512, (M, K, N, bits, p)
                        assert p["smem"] + 77 * 1024 > 228 * 1024 - 2048, (M, K, N, bits, p)
                        if bits == 4:
                            assert p["stages_w"] <= p["stages"] and p["stages_w"] >= 2 and p["stages_p"] >= 2
                            assert p["stages_p"] % 2 == 0 or p["stages_p"] >= p["stages_w"] + 2 or p["slot_first"]


@pytest.mark.parametrize("device", WHOLE + [(16, 8, 0, 0)])
def test_every_token_count_has_a_plan_that_fits(plans, device):
    """Each tile height there is, 16 to 256 tokens, with the last token of a tile and the first of the next one."""
    for bits in (4, 8):
        for K in (2048, 5120, 8192, 10496, 16384):
            for N in (1024, 2048, 2560, 4096, 6400, 8192):
                for M in [m for t in range(16, 1041, 16) for m in (t - 15, t - 1, t, t + 1)]:
                    p = plans.gemm(M, K, N, bits, device=device)
                    assert p["fits"] and p["smem"] <= 227 * 1024 and p["tmem_cols"] <= 512, (M, K, N, bits, p)


def test_ctas_of_a_pair_meet_between_their_last_read_of_tensor_memory_and_its_deallocation():
    """A pair's allocation is given back by both CTAs together: whatever else the kernel's end does, a barrier of the whole cluster,
    arrival and wait, lies between the outputs and the deallocation.  Its aligned arrivals are made by converged warps."""
    with open(os.path.join(CSRC, "gemm_tcgen05.cu")) as f:
        kernel = f.read().split("gemm_tcgen05_kernel(", 1)[1].split("// ---- host side", 1)[0]
    end = [line.split("//")[0].strip() for line in kernel[kernel.rindex("emit("):kernel.index("tmem_dealloc<CTAS>")].splitlines()]
    assert "if (CTAS == 2) cluster_sync_all();" in end and end.index("__syncthreads();") < end.index("if (CTAS == 2) cluster_sync_all();")
    lines = [line.split("//")[0].strip() for line in kernel.splitlines()]
    lines = [line for line in lines if line]
    assert lines[lines.index("cluster_arrive();") - 1] == "__syncwarp();" == lines[lines.index("if (CTAS == 1) cluster_arrive_relaxed();") - 1]


def route(plans, M, K, N, bits, device=None):
    """What runs the integer product of a call: the streaming kernel, a stacked tile, else how K is split."""
    p = plans.gemm(M, K, N, bits, device=device)
    assert p["fits"] and p["smem"] <= 227 * 1024 and p["tmem_cols"] <= 512, (M, K, N, bits, p)
    if p["stream"]:
        return "stream"
    if p["stack"] > 1:
        # one tile per CTA, and no second one behind it
        assert p["split"] == 1 and p["ctas"] == 1 and p["bt"] <= 128 and M <= p["bt"] // p["stack"] and N <= 64 * (device or plans.device)[0]
        return "stacked, %d atoms" % p["atoms"]
    return "%d %s" % (p["split"], "by clusters" if p["cluster"] else "tiles") if p["split"] > 1 else "tiles"


def test_stacked_tiles_and_their_lines(plans):
    call = lambda M, K, N, bits=4, device=None: route(plans, M, K, N, bits, device)
    assert [call(*c)[-7:] for c in edges.STACKED] == ["4 atoms"] * 4 + ["2 atoms"] * 2
    for inside, outside in [((32, 3072, 2048), (32, 2816, 2048)), ((32, 4096, 2048), (32, 4096, 2040)), ((32, 4096, 8704), (32, 4096, 8712)),
                            ((32, 6144, 4096), (32, 6144, 4088)), ((16, 16384, 5120), (16, 16384, 5112)), ((32, 8192, 9472), (32, 8192, 9480)),
                            ((48, 6144, 4608), (49, 6144, 4608)), ((64, 4096, 7168), (64, 4096, 7176)), ((64, 4096, 3072), (65, 4096, 3072)),
                            ((5, 4096, 8192), (4, 4096, 8192)), ((4, 4096, 7168), (2, 4096, 7168)), ((1, 7168, 7168), (1, 6912, 7168)),
                            ((1, 7168, 7168), (1, 7168, 7176)), ((2, 8192, 8192), (2, 8192, 8200)), ((1, 3072, 6144), (1, 3072, 6152))]:
        assert call(*inside).startswith("stacked") and not call(*outside).startswith("stacked"), (inside, outside)
    for M in (1, 4, 5, 16, 17, 32, 33, 48, 49, 64):
        for K in (3072, 3328, 4096, 8448, 16384):
            for N in (8, 136, 2048, 4744, 7168, 8704, 9472):
                for sms in (16, 148):
                    assert not call(M, K, N, 8, (sms, 74, 33, 14)).startswith("stacked")
                    got = call(M, K, N, 4, (sms, 74, 33, 14))
                    assert M > 4 or N <= 32 * sms or N > 64 * sms or got == "stream" or got.startswith("stacked"), (M, K, N, sms, got)


@pytest.mark.parametrize("device", WHOLE)
def test_sizes_of_the_parity_tests_take_the_routes_they_stand_for(plans, device):
    assert all(route(plans, M, K, N, 8, device) == "stream" for M, N, K in parity.STREAM_W8)
    assert route(plans, 16, 16384, 4096, 8, device) == "4 by clusters"
    assert all(route(plans, *c, device) == "stream" for c in parity.REPEATED_STREAM)
    assert all(route(plans, *c, device).startswith("stacked") for c in parity.REPEATED_STACKED)
    assert all(route(plans, *c, device).endswith("by clusters") for c in parity.REPEATED_CLUSTERS)
    assert all(route(plans, *c, device) == "tiles" for c in parity.REPEATED_TILES)
    sweep = {(M, KN, bits): route(plans, M, KN, KN, bits, device) for M, KN, _, bits in parity.SWEEP_SAMPLE}
    assert all(sweep[c] == "stream" for c in [(4, 6144, 4), (16, 4096, 4), (3, 1024, 8), (16, 4096, 8), (9, 2048, 8)])
    assert all(sweep[c].startswith("stacked") for c in [(8, 8192, 4), (16, 8192, 4)])
    assert all(route(plans, 16, K, N, bits, device) == "stream" for K, N, bits in [(4096, 4096, 4), (4096, 4096, 8), (8192, 1024, 4), (1024, 4096, 8)])


@pytest.mark.parametrize("device", WHOLE + [(148, 16, 0, 0)])
def test_short_batches_on_long_rows_leave_the_streaming_kernel_for_enough_slices_only(plans, device):
    """Every width from 9216 to 16384 channels: a call that the streaming kernel could take (one round of row groups, at most 64 Mi
    weights) runs there, or in clusters of four slices and more.  Without clusters of four it always runs there."""
    left = set()
    for bits in (4, 8):
        for K in range(9216, 16385, 256 if bits == 4 else 128):
            for M in (1, 8, 9, 12, 13, 16):
                for N in (8, 512, 1024, 1032, 2048, 4096, 4104, 4736):
                    if N * K > 1 << 26:
                        continue
                    got = route(plans, M, K, N, bits, device)
                    if got != "stream":
                        assert device[2] and got in ("4 by clusters", "8 by clusters") and K >= 10240, (M, K, N, bits, got)
                        assert M > 8 or (bits == 8 and N <= 1024 and got[0] == "8"), (M, K, N, bits, got)
                        left.add((M, K, N, bits))
    if device[2]:
        assert {(16, 10240, 2048, 4), (16, 16384, 4096, 4), (12, 12288, 4096, 4), (9, 10240, 2048, 8), (16, 10752, 2048, 8),
                (1, 10240, 1024, 8), (8, 16384, 512, 8)} <= left
    for M, K, N, bits in [(16, 9984, 2048, 4), (16, 10496, 4096, 4), (16, 10752, 4096, 4), (12, 10240, 2048, 4), (8, 16384, 1024, 4),
                          (1, 10368, 1024, 8), (8, 14464, 512, 8), (16, 16256, 4096, 8), (16, 10496, 4096, 8), (8, 16384, 1032, 8), (8, 10752, 512, 8)]:
        assert route(plans, M, K, N, bits, device) == "stream", (M, K, N, bits)
