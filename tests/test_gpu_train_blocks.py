"""Training form where the key side's CTAs take groups of blocks: full groups and a shorter last
one, several sequences, each block size and row size, against the fp64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from gpu_harness import h64, rel_l2
from test_gpu_train import TOL, TW, inputs, run_gpu

pytestmark = pytest.mark.gpu

# the group size follows the number of blocks: 1 while they fit the SMs, then the least waves
CASES = [
    TW("b16_groups_of_6", 40, 272, 4, 2, 64, 128, 16, 81),     # 17 blocks of 16: 6 + 6 + 5
    TW("b16_groups_of_8", 50, 384, 2, 1, 64, 64, 16, 85),      # 24 blocks: 8 + 8 + 8
    TW("b32_groups_of_4", 19, 416, 4, 2, 128, 128, 32, 82),    # 13 blocks of 32: 4 + 4 + 4 + 1
    TW("b64_groups_of_2", 36, 320, 2, 1, 128, 64, 64, 83),     # 5 blocks of 64: 2 + 2 + 1
    TW("b32_ungrouped", 3, 224, 2, 2, 64, 64, 32, 84),         # 42 blocks in all
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
