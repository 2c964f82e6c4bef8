"""The work that a user of this library has it do, as cases that can be timed.

A case is a dict of plain values; its "path" says which public entry points it goes through:

    linear      one projection, fq.linear: prologue + integer GEMM + epilogue in one call
    layer       the four projection sites of a language-backbone layer, one call each
    expert      one denoising step of the action expert: every site of every layer, replayed as one CUDA graph
    shared      one activation site with several consumers: fq.quantize_act once, fq.gemm_* per consumer
    gated       down_proj on the gate product: fq.linear_gated
    composite   a site with a stored composite rotation: fq.quantize_act_composite, then fq.gemm_*
    modulation  the weight-only projections of the adaptive layer norms of one step, replayed as one CUDA graph
    wonly       one weight-only projection of float activations, fq.linear_w4a16
    gptq        the offline fold of a 4-bit site with GPTQ rounding: fq.fold_weights_gptq and the export of its codes

Activations are Gaussian with a small share of outlier channels (the structure the method is made for), weights are
N(0, 0.02^2).  Sizes are those of the repository's own workloads (single linear, backbone layer, action expert,
throughput sweep, weight-only and GPTQ workloads) or generic ones.
"""
import math

import torch

from paper_2609_24433_b200 import fq

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}


# ---------------------------------------------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest call in earnest: one projection in binary32 with smoothing, called eagerly (launches and host time)
        {"name": "single_f32", "path": "linear", "M": 64, "K": 1024, "N": 1024, "block": 128, "bits": 4, "x": "f32", "y": "f32",
         "smooth": True, "clip": 1.0},
        # decode-sized batch on a large matrix: the 4-bit weights have to stream from memory once
        {"name": "short_w4", "path": "linear", "M": 16, "K": 8192, "N": 8192, "block": 64, "bits": 4, "x": "bf16", "y": "bf16",
         "smooth": False, "clip": 1.0},
        # the same regime with 8-bit weights, a few dozen tokens
        {"name": "short_w8", "path": "linear", "M": 64, "K": 8192, "N": 8192, "block": 64, "bits": 8, "x": "bf16", "y": "bf16",
         "smooth": False, "clip": 1.0},
        # a mid-sized prefill with nothing round about it: ragged tokens, ragged channels, a clip ratio below one
        {"name": "ragged_w8", "path": "linear", "M": 1000, "K": 4096, "N": 4104, "block": 128, "bits": 8, "x": "bf16", "y": "bf16",
         "smooth": True, "clip": 0.9},
        # the largest: a long batch, W4A4
        {"name": "long_w4", "path": "linear", "M": 16384, "K": 8192, "N": 8192, "block": 128, "bits": 4, "x": "bf16", "y": "bf16",
         "smooth": False, "clip": 1.0},
        # prefill of one language-backbone layer: 3 x 256 image + 48 text tokens, o_proj and down_proj at 8 bits
        {"name": "backbone_layer", "path": "layer", "M": 816, "hidden": 2048, "kv": 256, "mlp": 16384, "int8": True},
        # one step of the action expert's denoising loop, 50 action tokens through 18 layers
        {"name": "expert_step", "path": "expert", "M": 50, "width": 1024, "mlp": 4096, "layers": 18, "block": 64},
        # q, k and v as separate consumers of one quantized activation
        {"name": "shared_qkv", "path": "shared", "M": 816, "K": 2048, "N": 2048, "kv": 256, "block": 128, "bits": 4, "x": "bf16",
         "y": "bf16"},
        # down_proj straight from the fused gate/up output of a gated MLP
        {"name": "gated_down", "path": "gated", "M": 816, "K": 16384, "N": 2048, "block": 256, "bits": 8, "act": "gelu"},
        # the optional stored rotation of a site
        {"name": "composite", "path": "composite", "M": 816, "K": 2048, "N": 2048, "block": 64, "bits": 4, "x": "bf16", "y": "bf16"},
        # scale/shift/gate projections of one conditioning vector, one per layer
        {"name": "modulation", "path": "modulation", "M": 1, "K": 1536, "N": 3072, "layers": 18},
        # folding one 4-bit site of the backbone from its calibration tokens (offline, but every site of a model pays it)
        {"name": "gptq_site", "path": "gptq", "N": 2560, "K": 2048, "Mc": 4096, "block": 128, "x": "bf16"},
    ]


def _log(rng, lo, hi, step=1):
    """A size spread over the logarithm of [lo, hi], a multiple of `step`."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return int(min(hi, max(lo, round(v / step) * step)))


def draw(rng):
    path = rng.choice(["linear"] * 5 + ["layer", "expert", "shared", "gated", "composite", "modulation", "wonly", "gptq"])
    block = rng.choice([32, 64, 128, 256])
    bits = rng.choice([4, 8])
    if path == "linear":
        # most widths are multiples of the usual tiles, some are only multiples of what the library asks for
        kstep = rng.choice([256, max(block, 32)])
        c = {"path": path, "M": _log(rng, 1, 16384), "K": _log(rng, 1024, 16384, kstep), "N": _log(rng, 256, 16384, rng.choice([8, 128])),
             "block": block, "bits": bits, "x": rng.choice(["bf16", "bf16", "bf16", "f32"]), "y": rng.choice(["bf16", "bf16", "bf16", "f32"]),
             "smooth": rng.random() < 0.5, "clip": rng.choice([1.0, 1.0, 0.9])}
        most = 16384 * 8192 * 8192
        if c["M"] * c["K"] * c["N"] > most:
            c["M"] = max(1, most // (c["K"] * c["N"]))
        return c
    if path == "layer":
        return {"path": path, "M": _log(rng, 64, 2048), "hidden": 2048, "kv": 256, "mlp": rng.choice([8192, 16384]),
                "int8": rng.random() < 0.6}
    if path == "expert":
        return {"path": path, "M": rng.randrange(8, 65), "width": 1024, "mlp": rng.choice([2048, 4096]), "layers": rng.randrange(6, 19),
                "block": rng.choice([64, 128])}
    if path == "shared":
        return {"path": path, "M": _log(rng, 16, 4096), "K": _log(rng, 1024, 4096, 256), "N": _log(rng, 512, 4096, 64), "kv": 256,
                "block": block, "bits": bits, "x": "bf16", "y": rng.choice(["bf16", "f32"])}
    if path == "gated":
        return {"path": path, "M": _log(rng, 16, 2048), "K": _log(rng, 2048, 16384, 256), "N": _log(rng, 1024, 4096, 128), "block": block,
                "bits": bits, "act": rng.choice(["silu", "gelu"])}
    if path == "composite":
        return {"path": path, "M": _log(rng, 16, 2048), "K": _log(rng, 1024, 4096, 256), "N": _log(rng, 1024, 4096, 128),
                "block": rng.choice([32, 64, 128]), "bits": bits, "x": rng.choice(["bf16", "f32"]), "y": "bf16"}
    if path == "modulation":
        return {"path": path, "M": rng.randrange(1, 9), "K": _log(rng, 512, 2048, 256), "N": _log(rng, 1024, 6144, 128),
                "layers": rng.randrange(6, 19)}
    if path == "wonly":
        return {"path": path, "M": rng.randrange(1, 17), "K": _log(rng, 1024, 16384, rng.choice([256, 256, 128])),
                "N": _log(rng, 1024, 16384, 8), "x": rng.choice(["bf16", "bf16", "f32"]), "y": rng.choice(["bf16", "f32"])}
    return {"path": path, "N": _log(rng, 512, 2560, 8), "K": _log(rng, 512, 2048, 128), "Mc": _log(rng, 512, 4096), "block": rng.choice([64, 128]),
            "x": "bf16"}


# ------------------------------------------------------------------------------------------------------- inputs
class _Draw:
    """Tensors from one seed, on the GPU."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed) & 0x7FFFFFFF)

    def normal(self, *shape):
        return torch.randn(*shape, generator=self.g, device="cuda", dtype=torch.float32)

    def acts(self, M, K, dtype, frac=0.005, gain=30.0, sigma=1.0):
        """N(0, 1) with max(8, frac K) outlier channels: heavy-tailed (Student-t, three degrees of freedom) times `gain`."""
        x = self.normal(M, K)
        n = min(K, max(8, int(round(frac * K))))
        ch = torch.randperm(K, generator=self.g, device="cuda")[:n]
        self.channels = ch
        x[:, ch] = gain * self.normal(M, n) * torch.rsqrt(self.normal(3, M, n).square().mean(0))
        return (sigma * x).to(dtype)

    def weights(self, N, K):
        return 0.02 * self.normal(N, K), 0.02 * self.normal(N)


def _site(d, N, K, block, bits, x=None, smooth=False):
    """Folded weights of one consumer (smoothing calibrated on the activations at hand, exponent 0.5)."""
    W, b = d.weights(N, K)
    s = fq.smooth_scale(fq.col_absmax(x), fq.col_absmax(W), 0.5) if smooth else None
    return fq.fold_weights(W, s, b, block, bits)


def _graph(call):
    """`call` recorded once as a CUDA graph: how a control loop replays the same step."""
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        call()
    torch.cuda.current_stream().wait_stream(side)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call()
    return g


def _layer_sites(c):
    """(name, K, N, block, bits, smoothing, share of outlier channels)"""
    if c["path"] == "layer":
        h, od = c["hidden"], 8 if c["int8"] else 4
        return [("qkv", h, h + 2 * c["kv"], 128, 4, True, 0.01), ("o", h, h, 128, od, False, 0.01),
                ("gate_up", h, 2 * c["mlp"], 128, 4, True, 0.01), ("down", c["mlp"], h, 256, od, False, 0.005)]
    w, b = c["width"], c["block"]
    return [("qkv", w, 3 * w, b, 4, False, 0.005), ("o", w, w, b, 4, False, 0.005),
            ("gate_up", w, 2 * c["mlp"], b, 4, False, 0.005), ("down", c["mlp"], w, b, 4, False, 0.005)]


def _rotation(d, K, block):
    """A permutation and one orthogonal matrix per block of channels (a random basis behind a normalised Hadamard matrix)."""
    perm = torch.randperm(K, generator=d.g, device="cuda").to(torch.int32)
    h = torch.ones(1, 1, device="cuda")
    while h.shape[0] < block:
        h = torch.cat([torch.cat([h, h], 1), torch.cat([h, -h], 1)], 0)
    q = torch.linalg.qr(d.normal(K // block, block, block))[0]
    return perm, torch.matmul(h / math.sqrt(block), q.transpose(1, 2)).contiguous()


def prepare(case, seed):
    c, d = case, _Draw(seed)
    path = c["path"]
    st = {"case": c}
    if path == "linear":
        x = d.acts(c["M"], c["K"], DTYPES[c["x"]])
        st.update(x=x, W=_site(d, c["N"], c["K"], c["block"], c["bits"], x, c["smooth"]))
    elif path == "layer":
        st["sites"] = []
        for _, K, N, block, bits, smooth, frac in _layer_sites(c):
            x = d.acts(c["M"], K, torch.bfloat16, frac)
            st["sites"].append((x, _site(d, N, K, block, bits, x, smooth)))
    elif path == "expert":
        # the step's buffers are the program's own: inputs, outputs and one workspace that the stream-ordered calls share
        sites = _layer_sites(c)
        sigma = 1.0 - 0.9 * (seed % 10) / 9.0            # the activations' scale drifts over the denoising steps
        ws = torch.empty(max(fq.workspace_bytes(c["M"], K, N, bits) for _, K, N, _, bits, _, _ in sites), dtype=torch.uint8, device="cuda")
        ys = [torch.empty(c["layers"], c["M"], N, dtype=torch.bfloat16, device="cuda") for _, _, N, _, _, _, _ in sites]
        calls = []
        for layer in range(c["layers"]):
            for (_, K, N, block, bits, _, frac), y in zip(sites, ys):
                x = d.acts(c["M"], K, torch.bfloat16, frac, 20.0, sigma)
                calls.append((x, _site(d, N, K, block, bits), y[layer]))

        def step():
            for x, W, y in calls:
                fq.linear(x, W, y=y, workspace=ws)
        st.update(calls=calls, ws=ws, ys=ys, graph=_graph(step))
    elif path == "shared":
        x = d.acts(c["M"], c["K"], DTYPES[c["x"]], 0.01)
        W, b = d.weights(c["N"] + 2 * c["kv"], c["K"])
        s = fq.smooth_scale(fq.col_absmax(x), fq.col_absmax(W), 0.5)     # one diagonal for all consumers of the site
        at = [0, c["N"], c["N"] + c["kv"], c["N"] + 2 * c["kv"]]
        st.update(x=x, Ws=[fq.fold_weights(W[i:j], s, b[i:j].clone(), c["block"], c["bits"]) for i, j in zip(at, at[1:])])
    elif path == "gated":
        st.update(x=d.acts(c["M"], 2 * c["K"], torch.bfloat16, 0.005, 5.0), W=_site(d, c["N"], c["K"], c["block"], c["bits"]),
                  act=fq.GATE_GELU_TANH if c["act"] == "gelu" else fq.GATE_SILU)
    elif path == "composite":
        perm, blocks = _rotation(d, c["K"], c["block"])
        W, b = d.weights(c["N"], c["K"])
        st.update(x=d.acts(c["M"], c["K"], DTYPES[c["x"]]), perm=perm, blocks=blocks,
                  W=fq.fold_weights_composite(W, None, b, perm, blocks, c["bits"]))
    elif path == "modulation":
        x = d.normal(c["M"], c["K"]).to(torch.bfloat16)
        Ws = [_site(d, c["N"], c["K"], 1, 4) for _ in range(c["layers"])]
        ys = torch.empty(c["layers"], c["M"], c["N"], dtype=torch.bfloat16, device="cuda")

        def step():
            for W, y in zip(Ws, ys):
                fq.linear_w4a16(x, W, y=y)
        st.update(x=x, Ws=Ws, ys=ys, graph=_graph(step))
    elif path == "wonly":
        st.update(x=d.normal(c["M"], c["K"]).to(DTYPES[c["x"]]), W=_site(d, c["N"], c["K"], 1, 4))
    else:
        W, b = d.weights(c["N"], c["K"])
        x = d.acts(c["Mc"], c["K"], DTYPES[c["x"]], 0.01)
        # calibration tokens of a site are correlated across channels: a low-rank part on top
        x = (x.float() + d.normal(c["Mc"], 32) @ d.normal(32, c["K"])).to(DTYPES[c["x"]])
        st.update(W=W, b=b, x=x, s=fq.smooth_scale(fq.col_absmax(x), fq.col_absmax(W), 0.5))
    return st


def run(st):
    c = st["case"]
    path = c["path"]
    if path == "linear":
        return fq.linear(st["x"], st["W"], c["clip"], out_dtype=DTYPES[c["y"]])
    if path == "layer":
        return [fq.linear(x, W, out_dtype=torch.bfloat16) for x, W in st["sites"]]
    if path in ("expert", "modulation"):
        st["graph"].replay()
        return st["ys"]
    if path == "shared":
        gemm = fq.gemm_w4a4 if c["bits"] == 4 else fq.gemm_w8a8
        codes, delta = fq.quantize_act(st["x"], st["Ws"][0], c["block"], c["bits"])
        return [codes, delta] + [gemm(codes, delta, W, out_dtype=DTYPES[c["y"]]) for W in st["Ws"]]
    if path == "gated":
        return fq.linear_gated(st["x"], st["act"], st["W"], out_dtype=torch.bfloat16)
    if path == "composite":
        gemm = fq.gemm_w4a4 if c["bits"] == 4 else fq.gemm_w8a8
        codes, delta = fq.quantize_act_composite(st["x"], st["W"], st["perm"], st["blocks"], c["bits"])
        return [codes, delta, gemm(codes, delta, st["W"], out_dtype=DTYPES[c["y"]])]
    if path == "wonly":
        return fq.linear_w4a16(st["x"], st["W"], out_dtype=DTYPES[c["y"]])
    W = fq.fold_weights_gptq(st["W"], st["s"], st["b"], st["x"], c["block"], 4, 0.01)
    return W.export()


# ------------------------------------------------------------------------------------------------ bytes and sums
def _size(name):
    return 2 if name == "bf16" else 4


def _linear_work(M, K, N, bits, xs, ys, smooth):
    """Activations in, weights and their scales and bias in, outputs out; the product, and the transform's butterflies."""
    return {"bytes": M * K * xs + N * K * bits // 8 + 8 * N + (4 * K if smooth else 0) + M * N * ys, "flops": 2 * M * N * K}


def _sum(parts):
    return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}


def work(case):
    c = case
    path = c["path"]
    if path == "linear":
        return _linear_work(c["M"], c["K"], c["N"], c["bits"], _size(c["x"]), _size(c["y"]), c["smooth"])
    if path in ("layer", "expert"):
        one = _sum([_linear_work(c["M"], K, N, bits, 2, 2, smooth) for _, K, N, _, bits, smooth, _ in _layer_sites(c)])
        n = c.get("layers", 1)
        return {k: n * v for k, v in one.items()}
    if path == "shared":
        w = _linear_work(c["M"], c["K"], c["N"] + 2 * c["kv"], c["bits"], _size(c["x"]), _size(c["y"]), True)
        w["bytes"] += c["M"] * c["K"] * c["bits"] // 8 + 4 * c["M"]          # the codes and steps are outputs too
        return w
    if path == "gated":
        w = _linear_work(c["M"], c["K"], c["N"], c["bits"], 4, 2, False)     # two bf16 inputs per channel
        return w
    if path == "composite":
        w = _linear_work(c["M"], c["K"], c["N"], c["bits"], _size(c["x"]), _size(c["y"]), False)
        w["bytes"] += c["M"] * c["K"] * c["bits"] // 8 + 4 * c["M"] + 4 * c["K"] * (c["block"] + 1)
        w["flops"] += 2 * c["M"] * c["K"] * c["block"]
        return w
    if path in ("modulation", "wonly"):
        n = c.get("layers", 1)
        M, K, N, ys = c["M"], c["K"], c["N"], _size(c.get("y", "bf16"))
        return {"bytes": n * (N * K // 2 + 8 * N + M * N * ys) + M * K * _size(c.get("x", "bf16")), "flops": n * 2 * M * N * K}
    N, K, Mc = c["N"], c["K"], c["Mc"]
    # the second moment (symmetric), its factor, the factor's inverse, and the sweep over every weight row
    return {"bytes": 4 * N * K + Mc * K * _size(c["x"]) + N * K // 2 + 16 * N + 8 * K,
            "flops": K * K * Mc + K ** 3 / 3 + K ** 3 / 3 + N * K * K}


def tolerance(case):
    c = case
    if c["path"] == "gptq":
        return "exact"              # codes and steps are integers' work in a fixed order: the same bits from anybody
    # Codes, steps and integer sums are exact by definition; only the rescale (one multiply, one fused multiply-add), the sum of
    # the weight-only products and the rounding of the outputs are free.  TOLERANCES holds about four times what was measured.
    kind = "wonly" if c["path"] in ("modulation", "wonly") else "int"
    return dict(TOLERANCES[kind, c.get("y", "bf16")])


# Measured against the same rescale and sums in 64 bits, rounded once to the output type: integer paths 4.6e-8 (binary32 outputs)
# and at most 2.7e-5 (bf16: a value in some ten thousand rounds the other way, by one unit in the last place); weight-only paths
# 3e-6 (binary32 activations and outputs) and 1.2e-4 (bf16).
TOLERANCES = {
    ("int", "f32"): {"rel": 2e-7, "max": 1e-6},
    ("int", "bf16"): {"rel": 1.2e-4, "max": 1.6e-2},
    ("wonly", "f32"): {"rel": 1.2e-5, "max": 5e-5},
    ("wonly", "bf16"): {"rel": 5e-4, "max": 1.6e-2},
}
