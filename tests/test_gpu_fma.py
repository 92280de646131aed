"""The CUDA-core kernels (float32 throughout) and the feature map (tensor cores for bf16
rows) at the edges of their tiles, against the fp64 oracle: one row, one token, remainders of the 16 / 32 / 64-row tiles and of the
32-token chunks, every F, both head sizes, and batches that take each row-tile size.
"""
import math

import numpy as np
import pytest
import torch

import oracle
from gpu_harness import Pair, assert_parity, h64
from paper_2608_06628_gb300 import hybrid as H
from paper_2608_06628_gb300 import workloads as wk

pytestmark = pytest.mark.gpu

BF16, F32 = torch.bfloat16, torch.float32


@pytest.fixture(scope="module", autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_06628_gb300 import build
    build.build()
    torch.cuda.set_device(0)


# (dtype, n, Hq, Hkv, d, F, B)
SHAPES = [
    (F32, 1, 1, 1, 64, 16, 1),
    (F32, 2, 2, 1, 128, 16, 17),
    (F32, 1, 3, 1, 64, 32, 33),
    (F32, 2, 2, 2, 64, 64, 64),
    (F32, 1, 4, 2, 64, 128, 65),
    (F32, 1, 2, 2, 64, 256, 100),
    (F32, 1, 2, 1, 128, 256, 128),
    (F32, 38, 4, 4, 128, 128, 64),      # 64-row tiles
    (F32, 76, 2, 2, 64, 64, 64),
    (F32, 80, 4, 2, 128, 256, 24),
    (BF16, 2, 6, 2, 128, 128, 48),      # G = 3: no tensor-core step
    (BF16, 1, 3, 1, 64, 32, 20),
    # split operands on the tensor cores: items of 128 rows, the last one partial, one row,
    # F < 64, more items than SMs
    (BF16, 2, 4, 1, 128, 128, 64),
    (BF16, 3, 2, 2, 128, 64, 24),
    (BF16, 40, 8, 2, 64, 32, 48),
    (BF16, 2, 8, 1, 64, 256, 40),
    (BF16, 1, 1, 1, 64, 16, 1),
    (BF16, 2, 2, 2, 128, 16, 128),
    (BF16, 1, 2, 1, 128, 256, 127),
    (BF16, 45, 8, 4, 128, 128, 20),
]


@pytest.mark.parametrize("dt,n,Hq,Hkv,d,F,B", SHAPES)
def test_step_and_commit(dt, n, Hq, Hkv, d, F, B):
    wl = wk.Workload("fma", dt, n, Hq, Hkv, d, F, B, 61)
    pair = Pair(wl)
    pair.build_prefixes(np.arange(n) % 3 * B)
    Q, K, V = wk.block_qkv(wl, "fma", pair.dev)
    got, want, _ = pair.step(Q, K, V)
    assert_parity(got, want, dt, "output", units="out")
    K2, V2 = wk.prefix_kv(wl, 9, pair.dev, n_tok=B + 5)
    pair.commit(K2, V2)
    S, z = pair.gpu_state()
    assert_parity(S, pair.S, dt, "state S", units="state")
    assert_parity(z, pair.z, dt, "state z", units="state")


@pytest.mark.parametrize("F,k_scale", [(128, 1.0), (256, 8.0), (32, 24.0)])
def test_split_step_limits(F, k_scale):
    """Saturated gates, large scores, an empty prefix and a bad state pointer on the split step."""
    wl = wk.Workload("split", BF16, 3, 8, 2, 128, F, 40, 62, k_scale=k_scale)
    pair = Pair(wl)
    pair.build_prefixes(np.array([80, 40, 40]))
    Q, K, V = wk.block_qkv(wl, "split", pair.dev)
    for a in (math.inf, -math.inf, 30.0, -30.0, 0.0):
        alpha = torch.full((wl.Hq,), a, dtype=torch.float32, device=pair.dev)
        got, want, _ = pair.step(Q, K, V, alpha)
        assert_parity(got, want, BF16, f"alpha={a}", units="out")
    ptrs = pair.ptrs.clone()
    ptrs[1] = 0
    O = torch.full_like(Q, 7.0)
    H.hybrid_block_attn(pair.cfg, Q, K, V, pair.W, pair.alpha, ptrs, wl.n_req, O)
    assert H.hybrid_check(check=False) == H.HYBRID_ERR_DEVICE
    assert torch.all(O[1] == 7.0)
    fresh = Pair(wl)
    got, want, _ = fresh.step(Q, K, V)
    assert_parity(got, want, BF16, "empty prefix", units="out")


@pytest.mark.parametrize("dt", [F32, BF16])
@pytest.mark.parametrize("d,F,nh,Hkv,n_rows", [(64, 16, 1, 1, 1), (128, 32, 6, 2, 17), (64, 64, 8, 4, 700),
                                               (128, 128, 16, 4, 1237), (128, 256, 4, 4, 301), (64, 256, 2, 1, 65),
                                               # several tensor-core tiles per CTA, W changing on the way
                                               (64, 256, 8, 4, 5000), (128, 64, 2, 2, 40000), (128, 128, 24, 2, 50)])
def test_feature_map(dt, d, F, nh, Hkv, n_rows):
    g = torch.Generator(device="cuda").manual_seed(d + F + n_rows)
    X = torch.randn((n_rows, nh, d), generator=g, device="cuda").to(dt)
    W = (torch.randn((Hkv, d, F), generator=g, device="cuda") / math.sqrt(d)).to(dt)
    cfg = H.make_cfg(d, F, nh, Hkv, 32, dt)
    Phi = torch.full((n_rows + 1, nh, 2 * F), 7.0, dtype=torch.float32, device="cuda")
    H.hybrid_feature_map(cfg, X, n_rows, nh, W, Phi)
    H.hybrid_check()
    assert_parity(h64(Phi[:n_rows]), oracle.load().feature_map(h64(X), h64(W)), F32, "phi")
    assert torch.all(Phi[n_rows] == 7.0)
