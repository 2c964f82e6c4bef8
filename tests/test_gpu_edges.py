"""GPU parity at the sizes where a kernel or a dispatch rule can go wrong: edges of tiles, remainders, the smallest
and the largest of each variant's range.  Same oracle and same bounds as test_gpu_parity.py.  That the sizes in the lists
below take the routes they stand for, on whole B200s, is checked without a device in test_host_rules.py."""
import os
import subprocess
import sys
import threading
import time

import numpy as np
import pytest
import torch

import oracle
from helpers import to_dev, to_np
from paper_2609_24433_b200 import fq, synth
from test_gpu_parity import assert_fused_stages, make_x

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _watchdog_clean():
    yield
    st, word = fq.device_status()
    assert st == fq.OK, f"device wait watchdog fired: {word:#x}"


@pytest.mark.parametrize("N,K,Mc,block", [
    (8, 32, 5, 32),            # one block of the sweep, less than a tile of the second moment
    (40, 160, 33, 32),         # ragged tiles, one token into the second stage
    (24, 1184, 64, 32),        # exactly eight rows per CTA of the factor kernel on 148 SMs
    (16, 1216, 96, 64),        # ... and one row more on some
    (16, 2176, 64, 128),       # the longest rows of the factor kernel
    (8, 2208, 64, 32),         # the shortest of the column kernels
])
def test_gptq_fold_at_the_edges_of_its_kernels(N, K, Mc, block):
    rng = np.random.default_rng(N + K)
    W = synth.draw_weights(rng, N, K)
    calib = (rng.standard_normal((Mc, 8)) @ rng.standard_normal((8, K)) + rng.standard_normal((Mc, K))).astype(np.float32)
    wc, ws, _ = oracle.fold_weights_gptq(W, "f32", None, block, calib, "f32", 0.01, 4)
    hc, hs, _, _ = fq.fold_weights_gptq(to_dev(W), None, None, to_dev(calib), block, 4, 0.01).export()
    assert np.array_equal(to_np(hs).view(np.uint32), ws.view(np.uint32))
    assert np.array_equal(to_np(hc), wc)


GATED = [
    (296, 2048, 32, 4, oracle.SILU),                   # the shortest batch of the streamed gated rows on 148 SMs
    (295, 2048, 128, 8, oracle.GELU_TANH),             # the longest of the register kernel
    (3, 8448, 256, 8, oracle.GELU_TANH),               # long rows are streamed at any batch size
]


@pytest.mark.parametrize("M,K,block,bits,act", GATED)
def test_gated_prologue_on_both_sides_of_its_rule(M, K, block, bits, act):
    rng = np.random.default_rng(M + K)
    gu = rng.standard_normal((M, 2 * K)).astype(np.float32)
    gu[:, :K] *= 4.0
    gu[:, 7:K:97] *= 40.0                              # outlier gates: the clamped ends of the exponential
    gu[0, :6] = [0.0, -0.0, 3e38, -3e38, 9e37, -9e37]  # ... and what a quarter of the denominator would overflow
    gu[0, K:K + 6] = [1.0, 1.0, 1e-37, 1e-37, 1e-37, 1e-37]
    gu = synth.as_dtype(gu, "bf16")
    want_codes, want_delta = oracle.quantize_act_gated(gu, "bf16", act, None, block, bits, 1.0)
    codes, delta = fq.quantize_act_gated(to_dev(gu, "bf16"), act, None, block, bits, 1.0)
    assert np.array_equal(to_np(delta).view(np.uint32), want_delta.view(np.uint32))
    assert np.array_equal(to_np(codes), want_codes)


ODD_RINGS = [              # packed rings of an odd length, shorter than the two unpack sets' look-ahead
    (64, 4096, 8192),      # 64-token tiles of four-atom stages: a ring of three, three TMEM slots
    (96, 4096, 16384),     # two-atom stages: a ring of five, five TMEM slots
    (128, 4096, 16384),    # ... four TMEM slots
    (80, 4096, 2048),      # K split by clusters of four
]


@pytest.mark.parametrize("M,K,N", ODD_RINGS)
def test_odd_packed_rings_return_the_same_bits(M, K, N):
    """400 launches on rotating weights (so that the copies come from memory and land out of order), all equal to the
    CUDA-core witness."""
    g = torch.Generator(device="cuda").manual_seed(3)
    hs = [fq.weights_import(torch.randint(0, 255, (N, K // 2), dtype=torch.uint8, device="cuda", generator=g),
                            torch.rand(N, device="cuda", generator=g) + 0.1, None, None, K, 64, 4) for _ in range(10)]
    x = torch.randn(M, K, device="cuda", generator=g).to(torch.bfloat16)
    codes, delta = fq.quantize_act(x, None, 64, 4)
    want = [fq.gemm_simt(codes, delta, h, torch.bfloat16) for h in hs]
    ws = torch.empty(fq.workspace_bytes(M, K, N, 4), dtype=torch.uint8, device="cuda")
    ys = [torch.empty(M, N, dtype=torch.bfloat16, device="cuda") for _ in hs]
    graph = torch.cuda.CUDAGraph()
    for _ in range(2):
        for h, y in zip(hs, ys):
            fq.linear_w4a4(x, h, y=y, workspace=ws)
    with torch.cuda.graph(graph):
        for h, y in zip(hs, ys):
            fq.linear_w4a4(x, h, y=y, workspace=ws)
    for _ in range(40):
        graph.replay()
        for y, w in zip(ys, want):
            assert torch.equal(y, w)


ONE_LAUNCH = [
    (1, 128, 8, 32, 4, "bf16", False, 1.0),            # one token, one slice, one CTA
    (16, 256, 136, 256, 8, "f32", True, 0.9),          # a block as wide as a slice
    (17, 640, 1032, 128, 4, "f32", True, 1.0),         # five units over four CTAs, a ragged channel tile
    (8, 1024, 3072, 64, 4, "bf16", True, 1.0),         # the most CTAs with few tokens
    (32, 1024, 3072, 1, 8, "bf16", False, 1.0),        # identity rotation; the last batch of sixteen lanes a token
    (24, 1024, 4096, 64, 4, "bf16", True, 1.0),        # the most CTAs with up to 32 tokens
    (33, 1024, 1024, 64, 4, "bf16", True, 1.0),        # the first of eight
    (50, 1792, 1032, 8, 4, "bf16", False, 0.8),        # two rounds; fourteen units over eight CTAs: one round in some slices
    (64, 1920, 520, 128, 8, "bf16", True, 1.0),        # ... fifteen
    (64, 2048, 1024, 128, 4, "f32", False, 1.0),       # the longest rows of more than 32 tokens
    (32, 4096, 1024, 256, 4, "f32", False, 1.0),       # the longest rows
    (50, 896, 1024, 64, 4, "bf16", False, 1.0),        # the widest outputs in clusters of eight
    (63, 512, 1536, 64, 8, "f32", False, 1.0),         # ... of four
    (40, 384, 136, 128, 8, "bf16", True, 0.9),         # the shortest rows of more than 32 tokens
]


@pytest.mark.parametrize("M,K,N,block,bits,dtype,smooth,clip", ONE_LAUNCH)
def test_one_launch_path_equals_prologue_and_gemm(M, K, N, block, bits, dtype, smooth, clip):
    """Codes and steps against the oracle, outputs against the two-call route, all bit for bit, three replays of a graph
    of two calls on one workspace included."""
    rng = np.random.default_rng(M + K + N)
    W = torch.from_numpy(synth.draw_weights(rng, N, K)).cuda()
    s = torch.from_numpy(np.exp(rng.uniform(-1, 1, K)).astype(np.float32)).cuda() if smooth else None
    h = fq.fold_weights(W, s, torch.randn(N, device="cuda"), block, bits)
    x = make_x(M, K, dtype, seed=M)
    x_dev = to_dev(x, dtype)
    want = oracle.quantize_act(x, dtype, to_np(h.export()[2]), block, bits, clip)
    for ydt in (torch.float32, torch.bfloat16):
        y = assert_fused_stages(x_dev, h, clip, ydt, *want)
    ws = torch.zeros(fq.workspace_bytes(M, K, N, bits), dtype=torch.uint8, device="cuda")
    x2, ya, yb = x_dev.flip(0).contiguous(), torch.empty_like(y), torch.empty_like(y)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        fq.linear(x_dev, h, clip, y=ya, workspace=ws)
        fq.linear(x2, h, clip, y=yb, workspace=ws)
    for _ in range(3):
        g.replay()
    assert torch.equal(ya, y) and torch.equal(yb, y.flip(0))


COMPOSITE = [
    (1, 64, 64, 4, "bf16", False, 0),                  # one token, one item, one CTA
    (17, 512, 16, 8, "f32", True, 0),                  # the smallest blocks, one token into the second tile
    (33, 768, 256, 4, "bf16", True, 0),                # blocks of four items, an uneven share of them
    (700, 1024, 32, 4, "bf16", True, 8),               # more CTAs than SMs, rows with a lead
    (20, 4096, 128, 8, "f32", False, 0),               # binary32 rows of which eight fit
    (9, 8192, 64, 4, "f32", False, 0),                 # ... and none: the two-kernel form
    (20, 4096, 128, 8, "bf16", False, 4),              # rows that are not 16-byte aligned
    (576, 2048, 64, 4, "bf16", False, 0),              # a device that holds 36 clusters of four: the most in one wave
    (577, 2048, 64, 4, "bf16", True, 0),               # ... and clusters of two
]


@pytest.mark.parametrize("M,K,beta,bits,dtype,smooth,lead", COMPOSITE)
def test_composite_prologue_at_the_edges_of_its_kernels(M, K, beta, bits, dtype, smooth, lead):
    rng = np.random.default_rng(M + K)
    perm, blocks = synth.composite_rotation(K, beta, seed=K)
    x = make_x(M, K, dtype, seed=M)
    g = np.exp(rng.uniform(-1, 1, K)).astype(np.float32) if smooth else None
    want_codes, want_delta = oracle.composite_quantize(x, dtype, g, perm, blocks, bits, 0.9)
    big = torch.zeros((M, K + 8), dtype=torch.bfloat16 if dtype == "bf16" else torch.float32, device="cuda")
    x_dev = big[:, lead:lead + K]
    x_dev.copy_(to_dev(x, dtype))
    codes, delta = fq.quantize_act_composite(x_dev, to_dev(g), to_dev(perm), to_dev(blocks), bits, 0.9)
    assert np.array_equal(to_np(delta).view(np.uint32), want_delta.view(np.uint32))
    assert np.array_equal(to_np(codes), want_codes)


CLUSTER_SPLIT = [
    (64, 16384, 2048, 4),      # clusters of four, four-atom stages
    (16, 16384, 4224, 8),      # one token chunk: one CTA of four finishes the tile
    (100, 16384, 256, 4),      # few tiles: clusters of eight, ragged last chunk
    (50, 16384, 1024, 8),
    (90, 8192, 520, 8),        # a ragged channel tile
    (208, 16384, 136, 4),      # the longest batch in two tiles of 112 tokens
    (250, 16384, 128, 8),
    (816, 16384, 2048, 8),     # CTA pairs, clusters of two pairs
    (790, 16384, 1960, 8),     # ... with ragged tokens and channels
    (900, 16384, 2048, 8),     # ... tiles of 240 tokens: fifteen chunks, the most that a pair stages beside a ring of four
    (240, 8192, 8192, 8),
]


@pytest.mark.parametrize("M,K,N,bits", CLUSTER_SPLIT)
def test_cluster_split_equals_the_second_witness(M, K, N, bits):
    """int32 sums, binary32 and bf16 outputs, without any scratch in the workspace, a second call right behind the first."""
    g = torch.Generator(device="cuda").manual_seed(M + N)
    codes_w = torch.randint(0, 256, (N, K * bits // 8), dtype=torch.uint8, device="cuda", generator=g)
    h = fq.weights_import(codes_w, torch.rand(N, device="cuda", generator=g) + 0.1, None, torch.randn(N, device="cuda", generator=g),
                          K, 64, bits)
    x = torch.randn(M, K, device="cuda", generator=g)
    codes, delta = fq.quantize_act(x, None, 64, bits)
    ws = torch.empty((M * K + 255) // 256 * 256 + (4 * M + 255) // 256 * 256, dtype=torch.uint8, device="cuda")
    assert torch.equal(fq.gemm_acc_i32(codes, h, workspace=ws), fq.gemm_simt(codes, None, h, raw_acc=True))
    for dt in (torch.float32, torch.bfloat16):
        want = fq.gemm_simt(codes, delta, h, dt)
        a, b = fq.linear(x, h, out_dtype=dt, workspace=ws), fq.linear(x, h, out_dtype=dt, workspace=ws)
        assert torch.equal(a, want) and torch.equal(b, want)


STACKED = [                # two K slices of 64 channels in one tile
    (5, 3072, 4744),       # the shortest rows, two rounds of the streaming kernel's row groups, a ragged channel tile
    (17, 3328, 2056),      # thirteen k-blocks per slice: a last stage of one
    (32, 8192, 9472),      # a tile per SM
    (30, 16384, 5120),     # two chunks of tokens, the last one ragged
    (48, 6144, 7168),      # three: an uneven share
    (64, 3328, 2504),      # the longest batch
]


@pytest.mark.parametrize("M,K,N", STACKED)
def test_stacked_tiles_equal_the_second_witness(M, K, N):
    """int32 sums, binary32 and bf16 outputs bit for bit, in a workspace of codes and steps only; a second call right behind the
    first, and twenty replays over rotating weights, whose copies come from memory."""
    g = torch.Generator(device="cuda").manual_seed(M + N)
    hs = [fq.weights_import(torch.randint(0, 256, (N, K // 2), dtype=torch.uint8, device="cuda", generator=g),
                            torch.rand(N, device="cuda", generator=g) + 0.1, None, torch.randn(N, device="cuda", generator=g), K, 64, 4)
          for _ in range(8)]
    h, x = hs[0], torch.randn(M, K, device="cuda", generator=g)
    codes, delta = fq.quantize_act(x, None, 64, 4)
    ws = torch.empty((M * K + 255) // 256 * 256 + (4 * M + 255) // 256 * 256, dtype=torch.uint8, device="cuda")
    assert torch.equal(fq.gemm_acc_i32(codes, h, workspace=ws), fq.gemm_simt(codes, None, h, raw_acc=True))
    for dt in (torch.float32, torch.bfloat16):
        want = fq.gemm_simt(codes, delta, h, dt)
        a, b = fq.linear(x, h, out_dtype=dt, workspace=ws), fq.linear(x, h, out_dtype=dt, workspace=ws)
        assert torch.equal(a, want) and torch.equal(b, want)
    want = [fq.gemm_simt(codes, delta, h, torch.bfloat16) for h in hs]
    ys = [torch.empty_like(w) for w in want]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for h, y in zip(hs, ys):
            fq.linear(x, h, y=y, workspace=ws)
    for _ in range(20):
        graph.replay()
        for y, w in zip(ys, want):
            assert torch.equal(y, w)


SCRATCH_SPLIT = [
    (75, 20480, 4624, 8),      # more tiles than the clusters that a device holds: slices meet in the workspace
    (17, 32768, 4640, 4),      # four-atom stages
    (1562, 32768, 704, 4),     # token tiles of 144, which clusters do not take
    (1181, 32768, 712, 8),     # CTA pairs
]


@pytest.mark.parametrize("M,K,N,bits", SCRATCH_SPLIT)
def test_scratch_split_equals_the_second_witness(M, K, N, bits):
    """Through a workspace whose scratch (counters included) holds anything, through one that has none, and on three streams
    with a workspace each."""
    g = torch.Generator(device="cuda").manual_seed(M + N)
    h = fq.weights_import(torch.randint(0, 256, (N, K * bits // 8), dtype=torch.uint8, device="cuda", generator=g),
                          torch.rand(N, device="cuda", generator=g) + 0.1, None, torch.randn(N, device="cuda", generator=g), K, 64, bits)
    xs = [torch.randn(M, K, device="cuda", generator=g) for _ in range(3)]
    full, base = fq.workspace_bytes(M, K, N, bits), (M * K + 255) // 256 * 256 + (4 * M + 255) // 256 * 256
    assert full > base
    wss = [torch.randint(0, 256, (full,), dtype=torch.uint8, device="cuda", generator=g) for _ in xs]
    codes = [fq.quantize_act(x, None, 64, bits) for x in xs]
    assert torch.equal(fq.gemm_acc_i32(codes[0][0], h, workspace=wss[0]), fq.gemm_simt(codes[0][0], None, h, raw_acc=True))
    for dt in (torch.float32, torch.bfloat16):
        want = [fq.gemm_simt(c, d, h, dt) for c, d in codes]
        assert torch.equal(fq.linear(xs[0], h, out_dtype=dt, workspace=wss[0][:base]), want[0])
        torch.cuda.synchronize()
        got = []
        for x, ws, st in zip(xs, wss, [torch.cuda.Stream() for _ in xs]):
            with torch.cuda.stream(st):
                got.append([fq.linear(x, h, out_dtype=dt, workspace=ws) for _ in range(3)])
        torch.cuda.synchronize()
        assert all(torch.equal(y, w) for ys, w in zip(got, want) for y in ys)


W4_PAIRS = [
    (9001, 4096, 4352),        # 1.6e11 multiplications: CTA pairs, a ragged last token tile
    (16001, 2048, 5128),       # the shortest K, the last pair with no channel for its odd CTA
    (40001, 8256, 496),        # channels past K in the last k-block, the last pair nearly full
]
W4_SINGLE = [(9000, 4096, 4336)]   # just short of 1.6e11: single CTAs


@pytest.mark.parametrize("M,K,N", W4_PAIRS + W4_SINGLE)
def test_long_w4_pairs_equal_the_second_witness(M, K, N):
    g = torch.Generator(device="cuda").manual_seed(M + N)
    codes_w = torch.randint(0, 256, (N, K // 2), dtype=torch.uint8, device="cuda", generator=g)
    h = fq.weights_import(codes_w, torch.rand(N, device="cuda", generator=g) + 0.1, None, torch.randn(N, device="cuda", generator=g),
                          K, 64, 4)
    codes = torch.randint(0, 256, (M, K // 2), dtype=torch.uint8, device="cuda", generator=g)
    delta = torch.rand(M, device="cuda", generator=g) + 0.1
    for dt in (torch.float32, torch.bfloat16):
        assert torch.equal(fq.gemm_w4a4(codes, delta, h, dt), fq.gemm_simt(codes, delta, h, dt))
    assert torch.equal(fq.gemm_acc_i32(codes, h), fq.gemm_simt(codes, None, h, raw_acc=True))


W8_EPILOGUE = [            # tokens, K, channels, epilogue warps: unsplit launches on 8-bit weights
    (112, 256, 136, 16),       # short rows, short tiles, one round
    (130, 1280, 264, 8),       # longer rows
    (390, 512, 4000, 16),      # tiles of 112 tokens
    (299, 256, 16400, 16),     # two rounds, short rows
    (450, 2304, 12296, 8),     # two rounds, longer rows
    (1000, 512, 4104, 16),     # CTA pairs in one round
    (501, 2304, 13000, 16),    # ... in two
    (816, 1280, 9000, 8),      # ... and the ring a stage longer without the eight warps more
    (2300, 512, 4104, 16),     # three, short rows
    (4090, 1280, 4104, 16),    # four
    (3001, 2304, 5000, 8),     # four, longer rows
]


@pytest.mark.parametrize("M,K,N,warps", W8_EPILOGUE)
def test_w8_epilogues_equal_the_second_witness(M, K, N, warps):
    g = torch.Generator(device="cuda").manual_seed(M + N)
    codes_w = torch.randint(0, 256, (N, K), dtype=torch.uint8, device="cuda", generator=g)
    h = fq.weights_import(codes_w, torch.rand(N, device="cuda", generator=g) + 0.1, None, torch.randn(N, device="cuda", generator=g),
                          K, 64, 8)
    codes = torch.randint(0, 256, (M, K), dtype=torch.uint8, device="cuda", generator=g)
    delta = torch.rand(M, device="cuda", generator=g) + 0.1
    for dt in (torch.float32, torch.bfloat16):
        assert torch.equal(fq.gemm_w8a8(codes, delta, h, dt), fq.gemm_simt(codes, delta, h, dt))
    assert torch.equal(fq.gemm_acc_i32(codes, h), fq.gemm_simt(codes, None, h, raw_acc=True))


FEW_UNITS = [
    (9, 1536, 256, 8),         # six units of K for clusters of eight
    (31, 1792, 256, 4),        # seven
    (33, 384, 64, 4),          # three for clusters of four
    (64, 896, 128, 8),
]


@pytest.mark.parametrize("M,K,block,bits", FEW_UNITS)
def test_one_launch_with_fewer_units_than_cluster_ctas(M, K, block, bits):
    """CTAs without channels add nothing, whatever the launch ahead left in tensor memory."""
    g = torch.Generator(device="cuda").manual_seed(K)
    h = fq.weights_import(torch.randint(0, 256, (200, K * bits // 8), dtype=torch.uint8, device="cuda", generator=g),
                          torch.rand(200, device="cuda", generator=g) + 0.1, None, None, K, block, bits)
    x, many = (torch.randn(m, K, device="cuda", generator=g) for m in (M, 4000))
    codes, delta = fq.quantize_act(x, None, block, bits)
    want = fq.gemm_simt(codes, delta, h, torch.float32)
    for _ in range(50):
        fq.linear(many, h)     # fills tensor memory with sums
        assert torch.equal(fq.linear(x, h), want)


PROLOGUE = [
    (1300, 2048, 128, 8, "bf16", "smooth"),            # 148 SMs: the longest batch of the register kernel
    (1301, 2048, 128, 8, "bf16", "smooth"),            # ... and the shortest streamed one
    (5607, 2112, 64, 4, "bf16", "plain"),              # one lane of the row's last warp has channels
    (269, 8256, 32, 8, "bf16", "plain"),               # warps without any
    (73, 16384, 256, 4, "bf16", "plain"),              # the longest rows, fewer than SMs
    (651, 4096, 128, 8, "bf16", "after"),              # 32 channels per thread
    (1735, 1536, 256, 4, "bf16", "smooth"),
    (558, 7168, 64, 4, "bf16", "plain"),               # seven eighths of the lanes
    (2168, 3072, 128, 8, "bf16", "smooth"),            # three quarters
    (7516, 2560, 128, 4, "bf16", "smooth"),            # less
    (217, 10240, 128, 8, "bf16", "smooth"),            # ... behind 8192 channels
    (1879, 1024, 64, 8, "f32", "smooth"),
    (145, 8192, 32, 4, "f32", "plain"),
    (868, 2560, 64, 8, "f32", "plain"),                # 64 channels per thread
    (3469, 2560, 128, 4, "f32", "smooth"),
    (538, 4128, 32, 8, "f32", "plain"),
]


@pytest.mark.parametrize("M,K,block,bits,dtype,form", PROLOGUE)
def test_streamed_prologue_on_both_sides_of_its_rule(M, K, block, bits, dtype, form):
    """Eight rows against the oracle, all of them against short batches, which never stream; codes as a caller sees them
    (packed or int8) and, through a small layer, as the GEMM reads them."""
    rng = np.random.default_rng(M + K)
    x = make_x(M, K, dtype, seed=M)
    mult = None if form == "plain" else np.exp(rng.uniform(-1, 1, K)).astype(np.float32)
    x_dev, m_dev, after, clip = to_dev(x, dtype), to_dev(mult), form == "after", 0.9 if bits == 8 else 1.0
    codes, delta = fq.quantize_act(x_dev, m_dev, block, bits, clip, fold_after=after)
    rows = rng.choice(M, 8, replace=False)
    quantize = oracle.quantize_act_after if after else oracle.quantize_act
    want_codes, want_delta = quantize(x[rows], dtype, mult, block, bits, clip)
    assert np.array_equal(to_np(delta)[rows].view(np.uint32), want_delta.view(np.uint32))
    assert np.array_equal(to_np(codes)[rows], want_codes)
    g = torch.Generator(device="cuda").manual_seed(K)
    h = fq.weights_import(torch.randint(0, 256, (16, K * bits // 8), dtype=torch.uint8, device="cuda", generator=g),
                          torch.rand(16, device="cuda", generator=g) + 0.1, m_dev, None, K, block, bits, fold_after=after)
    y = fq.linear(x_dev, h, clip)
    for r in range(0, M, 40):
        part = x_dev[r:r + 40]
        c, d = fq.quantize_act(part, m_dev, block, bits, clip, fold_after=after)
        assert torch.equal(c, codes[r:r + 40]) and torch.equal(d, delta[r:r + 40])
        assert torch.equal(fq.linear(part, h, clip), y[r:r + 40])


@pytest.mark.parametrize("act", [-1, -7, 2, 1 << 32, (1 << 32) + 1])
def test_linear_gated_refuses_what_is_no_gate(act):
    """No number but the two functions' own is a gate: not one that could stand for "ungated", nor one that is narrowed."""
    h = fq.fold_weights(torch.randn(16, 64, device="cuda"), None, None, 32, 4)
    gate_up = torch.randn(4, 128, device="cuda")
    with pytest.raises(fq.FqError) as e:
        fq.linear_gated(gate_up, act, h)
    assert e.value.status == fq.ERR_INVALID_ARG


TO_AND_FRO = [
    (50, 1024, 4, "linear"),           # one launch a call
    (64, 1024, 8, "linear"),
    (5, 768, 4, "linear"),
    (24, 4096, 4, "linear"),           # prologue and GEMM
    (12, 4096, 8, "linear"),           # prologue and weight streaming
    (300, 1024, 4, "linear"),
    (2, 1536, 4, "linear_w4a16"),
]


@pytest.mark.parametrize("M,K,bits,call", TO_AND_FRO)
def test_calls_that_pass_two_buffers_to_and_fro(M, K, bits, call):
    """A -> B, B -> A, A -> B ...: kernels of three calls are resident at a time, and the third reads what the second wrote over the
    first one's input.  As a graph and eagerly, against the same calls with a synchronisation behind each."""
    g = torch.Generator(device="cuda").manual_seed(M + K)
    hs = [fq.weights_import(torch.randint(0, 256, (K, K * bits // 8), dtype=torch.uint8, device="cuda", generator=g),
                            (torch.rand(K, device="cuda", generator=g) + 0.5) / (0.3 * K ** 0.5 * (5 if bits == 4 else 74)), None,
                            torch.randn(K, device="cuda", generator=g), K, 64 if call == "linear" else 1, bits) for _ in range(3)]
    ws = torch.empty(fq.workspace_bytes(M, K, K, bits), dtype=torch.uint8, device="cuda")
    a, b = (torch.empty(M, K, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    start = torch.randn(M, K, device="cuda", generator=g).to(torch.bfloat16)

    def chain(sync=False):
        a.copy_(start)
        x, y = a, b
        for step in range(13):
            if call == "linear":
                fq.linear(x, hs[step % 3], y=y, workspace=ws)
            else:
                fq.linear_w4a16(x, hs[step % 3], y=y)
            if sync:
                torch.cuda.synchronize()
            x, y = y, x

    chain(sync=True)
    want = a.clone(), b.clone()
    assert all(w.isfinite().all() and w.float().std() > 0.1 for w in want)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        chain()
    for run in [graph.replay] * 40 + [chain] * 10:
        a.fill_(7.0), b.fill_(7.0)
        run()
        assert torch.equal(a, want[0]) and torch.equal(b, want[1])


FIRST_CALLS = """
import ctypes, sys, threading
import torch
from paper_2609_24433_b200 import fq
torch.cuda.init()
shapes = [(8, 256, 64), (24, 512, 128), (50, 1024, 64), (64, 2048, 64), (200, 1024, 128), (700, 2048, 128), (16, 4096, 256), (40, 1536, 128)]
Ws = [torch.randn(N, K, device="cuda") for _, K, N in shapes]
xs = [torch.randn(M, K, device="cuda") for M, K, _ in shapes]
torch.cuda.synchronize()
gate, errors, ys = threading.Barrier(len(shapes)), [], [None] * len(shapes)

def work(i):
    try:
        gate.wait()
        with torch.cuda.stream(torch.cuda.Stream()):
            h = fq.fold_weights(Ws[i], None, None, 32, 4)          # the first calls of the process: folds and projections
            for _ in range(20):
                ys[i] = fq.linear(xs[i], h)
            torch.cuda.current_stream().synchronize()
    except Exception as e:
        errors.append((i, repr(e)))

threads = [threading.Thread(target=work, args=(i,)) for i in range(len(shapes))]
[t.start() for t in threads]
[t.join() for t in threads]
assert not errors, errors
for W, x, y in zip(Ws, xs, ys):
    assert torch.equal(y, fq.linear(x, fq.fold_weights(W, None, None, 32, 4)))
assert fq.device_status()[0] == fq.OK
"""


def test_first_calls_of_a_process_from_several_threads():
    """What is looked up once (driver entry point, kernel attributes, device facts) is looked up by eight threads at a time."""
    r = subprocess.run([sys.executable, "-c", FIRST_CALLS], cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]


@pytest.mark.parametrize("call", ["linear", "gemm", "quantize_act", "linear_w4a16", "linear_gated", "quantize_act_composite"])
def test_other_python_threads_run_while_a_launch_waits(call):
    """Launches behind a busy stream wait once its queue is full; a second thread keeps counting all the while."""
    h, x = fq.fold_weights(torch.randn(64, 256, device="cuda"), None, None, 1, 4), torch.randn(8, 256, device="cuda")
    gate_up, ws = torch.randn(8, 512, device="cuda"), torch.empty(1 << 16, dtype=torch.uint8, device="cuda")
    perm, blocks = (to_dev(a) for a in synth.composite_rotation(256, 32, seed=1))
    codes, delta = fq.quantize_act(x, None, 1, 4)
    y = torch.empty(8, 64, device="cuda")
    run = {"linear": lambda: fq.linear(x, h, y=y, workspace=ws), "gemm": lambda: fq.gemm_w4a4(codes, delta, h, y=y, workspace=ws),
           "quantize_act": lambda: fq.quantize_act(x, None, 1, 4, codes=codes, delta=delta),
           "linear_w4a16": lambda: fq.linear_w4a16(x, h, y=y), "linear_gated": lambda: fq.linear_gated(gate_up, fq.GATE_SILU, h, y=y, workspace=ws),
           "quantize_act_composite": lambda: fq.quantize_act_composite(x, None, perm, blocks, 4, codes=codes, delta=delta, workspace=ws)}[call]
    run()
    torch.cuda.synchronize()
    for _ in range(5):                                    # (again where the host was held up until the stream was idle)
        done, ticks = threading.Event(), []

        def count():
            while not done.wait(0.002):
                ticks.append(time.perf_counter())

        torch.cuda._sleep(int(0.8 * 1.9e9))               # the stream is busy for 0.8 s or a little more
        thread = threading.Thread(target=count)
        thread.start()
        longest, start = 0.0, time.perf_counter()
        while longest < 0.2 and time.perf_counter() < start + 0.6:
            t = time.perf_counter()
            run()
            longest = max(longest, time.perf_counter() - t)
        done.set()
        thread.join()
        gaps = np.diff([start] + ticks)
        torch.cuda.synchronize()
        if longest > 0.2:
            break
    assert longest > 0.2, f"no launch had to wait ({longest:.3f} s): nothing was tested"
    assert gaps.max() < 0.5 * longest, f"a launch waited {longest:.3f} s, the other thread stood still for {gaps.max():.3f} s"
