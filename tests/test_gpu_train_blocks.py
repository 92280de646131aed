"""Training form where the key side's CTAs take groups of blocks: full groups and a shorter last
one, several sequences, each block size and row size, against the fp64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from gpu_harness import h64, rel_l2
from test_gpu_train import TOL, TW, inputs, run_gpu

pytestmark = pytest.mark.gpu

CASES = [
    TW("b16_17_blocks", 2, 272, 4, 2, 64, 128, 16, 81),    # 8 + 8 + 1 blocks of 16
    TW("b32_9_blocks", 2, 288, 8, 2, 128, 128, 32, 82),    # 4 + 4 + 1
    TW("b64_5_blocks", 2, 320, 2, 1, 128, 64, 64, 83),     # 2 + 2 + 1
    TW("b32_7_blocks", 3, 224, 2, 2, 64, 64, 32, 84),      # 4 + 3
]


@pytest.mark.parametrize("wl", CASES, ids=[w.name for w in CASES])
def test_block_groups(wl):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_06628_gb300 import build
    build.build()
    Q, K, V, W, alpha, dO = inputs(wl)
    O, dW, dalpha = run_gpu(wl, Q, K, V, W, alpha, dO)
    orc = oracle.load()
    args = (h64(Q), h64(K), h64(V), h64(W), h64(alpha))
    dW_ref, da_ref = orc.train_backward(*args, h64(dO), wl.B)
    for got, want, what in ((O, orc.train_forward(*args, wl.B), "O"), (dW, dW_ref, "dW"), (dalpha, da_ref, "dalpha")):
        g = h64(got)
        assert np.all(np.isfinite(g)), what
        assert rel_l2(g, want) <= TOL, what
