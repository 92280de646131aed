"""Step and commit in one pass for F = 256 against the fp64 oracle: one unit, several units
per CTA, every group size that fits 64 query rows, blocks shorter than the 64-row tile,
large scores, saturated gates, an empty prefix and a bad state pointer."""
import math

import numpy as np
import pytest
import torch

from gpu_harness import Pair, assert_parity, h64
from paper_2608_06628_gb300 import hybrid as H
from paper_2608_06628_gb300 import workloads as wk

pytestmark = pytest.mark.gpu

BF16 = torch.bfloat16


@pytest.fixture(scope="module", autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_06628_gb300 import build
    build.build()
    torch.cuda.set_device(0)


def fused(pair, Q, K, V, alpha=None, ptrs=None):
    """Runs the fused call; the oracle's output and committed state beside it."""
    alpha = pair.alpha if alpha is None else alpha
    O = torch.full_like(Q, 7.0)
    H.hybrid_block_attn_commit(pair.cfg, Q, K, V, pair.W, alpha, pair.ptrs if ptrs is None else ptrs, pair.wl.n_req, O)
    want = pair.orc.block_attn(h64(Q), h64(K), h64(V), pair.W64, h64(alpha), pair.S, pair.z)
    pair.orc.commit(h64(K), h64(V), pair.W64, pair.S, pair.z)
    return O, want


# (n, Hq, Hkv, d, B, k_scale)
@pytest.mark.parametrize("n,Hq,Hkv,d,B,k_scale", [
    (1, 1, 1, 128, 64, 1.0), (3, 2, 2, 128, 64, 8.0), (2, 8, 2, 128, 16, 1.0), (5, 4, 2, 64, 32, 1.0),
    (2, 3, 3, 128, 48, 8.0), (1, 4, 1, 64, 16, 24.0), (41, 8, 8, 64, 16, 1.0), (40, 16, 8, 128, 32, 1.0)])
def test_two_blocks(n, Hq, Hkv, d, B, k_scale):
    wl = wk.Workload("wide", BF16, n, Hq, Hkv, d, 256, B, 63, k_scale=k_scale)
    pair = Pair(wl)
    pair.build_prefixes(np.arange(n) % 3 * B)
    for tag in ("a", "b"):
        Q, K, V = wk.block_qkv(wl, tag, pair.dev)
        O, want = fused(pair, Q, K, V)
        H.hybrid_check()
        assert_parity(h64(O), want, BF16, "output", units="out")
        S, z = pair.gpu_state()
        assert_parity(S, pair.S, BF16, "state S", units="state")
        assert_parity(z, pair.z, BF16, "state z", units="state")


def test_gates_and_bad_pointer():
    wl = wk.Workload("wide", BF16, 3, 4, 2, 128, 256, 32, 64, k_scale=8.0)
    pair = Pair(wl)
    pair.build_prefixes(np.array([64, 32, 32]))
    for i, al in enumerate((math.inf, -math.inf, 30.0, -30.0)):
        Q, K, V = wk.block_qkv(wl, i, pair.dev)
        O, want = fused(pair, Q, K, V, torch.full((wl.Hq,), al, dtype=torch.float32, device=pair.dev))
        H.hybrid_check()
        assert_parity(h64(O), want, BF16, f"alpha={al}", units="out")
    before = pair.pool.slab.clone().view(3, -1)
    ptrs = pair.ptrs.clone()
    ptrs[1] = 8                       # misaligned: reported, its request skipped
    O, want = fused(pair, Q, K, V, ptrs=ptrs)
    assert H.hybrid_check(check=False) == H.HYBRID_ERR_DEVICE
    assert torch.all(O[1] == 7.0) and torch.equal(pair.pool.slab.view(3, -1)[1], before[1])
    assert_parity(h64(O)[[0, 2]], want[[0, 2]], BF16, "others", units="out")
    S, z = pair.gpu_state()
    assert_parity(S[[0, 2]], pair.S[[0, 2]], BF16, "others' S", units="state")
    fresh = Pair(wl)
    O, want = fused(fresh, Q, K, V)
    H.hybrid_check()
    assert_parity(h64(O), want, BF16, "empty prefix", units="out")
