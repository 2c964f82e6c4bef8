"""GPU parity at the sizes where a kernel or a dispatch rule can go wrong: edges of tiles, remainders, the smallest
and the largest of each variant's range.  Same oracle and same bounds as test_gpu_parity.py."""
import numpy as np
import pytest
import torch

import oracle
from helpers import to_dev, to_np
from paper_2609_24433_b200 import fq, synth

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
