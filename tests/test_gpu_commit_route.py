"""Commits of at most a block's tokens on both sides of the choice between the two tensor-core
kernels (one wave of units or none, more than three, 32 tokens and one more), uniform and ragged,
against the fp64 oracle."""
import numpy as np
import pytest
import torch

from gpu_harness import Pair, assert_parity, h64
from paper_2608_06628_gb300 import hybrid as H
from paper_2608_06628_gb300 import workloads as wk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,Hkv,d,F,T", [
    (19, 4, 128, 128, 32), (20, 4, 128, 128, 32), (114, 4, 128, 128, 17), (115, 4, 128, 128, 32),
    (40, 4, 128, 128, 33), (40, 4, 128, 128, 64), (40, 4, 64, 128, 32), (40, 4, 128, 64, 1), (200, 2, 64, 64, 48),
])
@pytest.mark.parametrize("ragged", [False, True])
def test_short_commit(n, Hkv, d, F, T, ragged):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_06628_gb300 import build
    build.build()
    wl = wk.Workload("route", torch.bfloat16, n, Hkv, Hkv, d, F, 32, 68)
    tracked = np.unique(np.r_[0:6, n - 6:n])
    pair = Pair(wl, tracked=tracked)
    K, V = wk.prefix_kv(wl, 74, pair.dev, n_tok=T)
    lens = np.array([T] + [(5 * r) % (T + 1) for r in range(1, n)]) if ragged else np.full(n, T)
    if ragged:
        Kp = torch.cat([K[r, :lens[r]] for r in range(n)]).contiguous()
        Vp = torch.cat([V[r, :lens[r]] for r in range(n)]).contiguous()
        offs = np.concatenate([[0], np.cumsum(lens)]).tolist()
        H.hybrid_commit_ragged(pair.cfg, Kp, Vp, offs, pair.W, pair.ptrs, n)
    else:
        H.hybrid_commit_block(pair.cfg, K, V, T, pair.W, pair.ptrs, n)
    H.hybrid_check()
    for i, r in enumerate(tracked):
        if lens[r]:
            S, z = pair.S[i:i + 1].copy(), pair.z[i:i + 1].copy()
            pair.orc.commit(h64(K[r:r + 1, :lens[r]]), h64(V[r:r + 1, :lens[r]]), pair.W64, S, z)
            pair.S[i:i + 1], pair.z[i:i + 1] = S, z
    S, z = pair.gpu_state()
    assert_parity(S, pair.S, torch.bfloat16, "state S", units="state")
    assert_parity(z, pair.z, torch.bfloat16, "state z", units="state")


def test_short_commit_repeats_bitwise():
    """64 tokens per request (two warps' token sums): the same bits from run to run."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_06628_gb300 import build
    build.build()
    wl = wk.Workload("repeat", torch.bfloat16, 400, 2, 2, 128, 128, 32, 69)
    K, V = wk.prefix_kv(wl, 75, "cuda", n_tok=64)
    slabs = []
    for _ in range(4):
        pair = Pair(wl, tracked=[0])
        H.hybrid_commit_block(pair.cfg, K, V, 64, pair.W, pair.ptrs, wl.n_req)
        H.hybrid_commit_block(pair.cfg, V[:, :40].contiguous(), K[:, :40].contiguous(), 40, pair.W, pair.ptrs, wl.n_req)
        H.hybrid_check()
        slabs.append(pair.pool.slab.clone())
    assert all(torch.equal(s, slabs[0]) for s in slabs)
