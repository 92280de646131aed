"""A commit folds each request's own tokens only: with NaN and infinity in every other request's
K and V and token counts that are no multiple of 16 (the depth of a tensor-core product), the
states of the requests between them are those of a commit without them."""
import numpy as np
import pytest
import torch

from gpu_harness import Pair
from paper_2608_06628_gb300 import hybrid as H
from paper_2608_06628_gb300 import workloads as wk

pytestmark = pytest.mark.gpu

BF16, F32 = torch.bfloat16, torch.float32


# (dtype, n, Hkv, d, F, T)
@pytest.mark.parametrize("dt,n,Hkv,d,F,T", [
    # token-major kernel, at most 64 tokens and more, one chunk of 128 and several
    (BF16, 200, 2, 64, 64, 40), (BF16, 40, 4, 128, 64, 17), (BF16, 8, 2, 128, 128, 1), (BF16, 9, 4, 64, 128, 63),
    (BF16, 40, 4, 128, 128, 100), (BF16, 6, 2, 64, 64, 130), (BF16, 7, 2, 128, 128, 265),
    # reduction kernel (d = F = 128 between half a wave and three waves; F = 256)
    (BF16, 30, 4, 128, 128, 24), (BF16, 30, 4, 128, 128, 31), (BF16, 6, 2, 128, 256, 24), (BF16, 7, 2, 64, 256, 45),
    # CUDA cores
    (BF16, 6, 2, 64, 32, 21), (F32, 6, 2, 64, 64, 21),
])
@pytest.mark.parametrize("ragged", [False, True])
def test_neighbours_do_not_leak(dt, n, Hkv, d, F, T, ragged):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_06628_gb300 import build
    build.build()
    wl = wk.Workload("isolation", dt, n, Hkv, Hkv, d, F, 32, 91)
    K, V = wk.prefix_kv(wl, 0, "cuda", n_tok=T)
    lens = np.full(n, T) if not ragged else np.maximum(1, T - np.arange(n) % 5)
    Kb, Vb = K.clone(), V.clone()
    Kb[1::2] = float("nan")
    Vb[1::4] = float("nan")
    Vb[3::4] = float("inf")

    def folded(K, V):
        pair = Pair(wl, tracked=[0])
        if ragged:
            Kp, Vp = (torch.cat([x[r, :lens[r]] for r in range(n)]).contiguous() for x in (K, V))
            H.hybrid_commit_ragged(pair.cfg, Kp, Vp, np.concatenate([[0], np.cumsum(lens)]).tolist(), pair.W, pair.ptrs, n)
        else:
            H.hybrid_commit_block(pair.cfg, K, V, T, pair.W, pair.ptrs, n)
        H.hybrid_check()
        return pair.pool.slab.clone().view(n, -1)

    clean, mixed = folded(K, V), folded(Kb, Vb)
    assert not torch.isfinite(mixed[1::2]).all(1).any()
    assert torch.isfinite(mixed[0::2]).all(1).all()
    # the increments of a unit's runs (at most T / 128 + 1 here) are added in any order: a few
    # float32 roundings of sums no larger than the state's largest element
    assert (mixed[0::2] - clean[0::2]).abs().max() <= 2.0 ** -20 * clean[0::2].abs().max()
