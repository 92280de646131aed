"""Prompts folded as many short runs per CTA (each run's sums leave beside the next run's
chunks), with empty prompts and unusable state pointers among them, against the fp64 oracle."""
import numpy as np
import pytest
import torch

from gpu_harness import Pair, assert_parity, h64
from paper_2608_06628_gb300 import hybrid as H
from paper_2608_06628_gb300 import workloads as wk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,F", [(128, 128), (128, 64), (64, 128), (64, 64)])
def test_short_runs(d, F):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_06628_gb300 import build
    build.build()
    n, Hkv = 250, 2
    wl = wk.Workload("runs", torch.bfloat16, n, 2, Hkv, d, F, 32, 66)
    pair = Pair(wl)
    pair.build_prefixes(np.arange(n) % 2 * 32)
    # one to three chunks each, full, one token over and one short; the first is the longest
    lens = np.array([300] + [[128, 1, 129, 0, 256, 40, 127, 33][r % 8] for r in range(1, n)])
    bad = np.array([r % 9 == 4 or r == n - 1 for r in range(n)])
    ptrs = pair.ptrs.clone()
    ptrs[torch.as_tensor(bad)] = 0
    before = pair.pool.slab.clone().view(n, -1)
    offs = np.concatenate([[0], np.cumsum(lens)])
    K, V = wk.prefix_kv(wl, 73, pair.dev, n_req=1, n_tok=int(offs[-1]))
    Kp, Vp = K[0].contiguous(), V[0].contiguous()
    H.hybrid_commit_ragged(pair.cfg, Kp, Vp, offs.tolist(), pair.W, ptrs, n)
    assert H.hybrid_check(check=False) == H.HYBRID_ERR_DEVICE
    for r in np.nonzero(~bad & (lens > 0))[0]:
        a, b = int(offs[r]), int(offs[r + 1])
        S, z = pair.S[r:r + 1].copy(), pair.z[r:r + 1].copy()
        pair.orc.commit(h64(Kp[a:b][None]), h64(Vp[a:b][None]), pair.W64, S, z)
        pair.S[r:r + 1], pair.z[r:r + 1] = S, z
    good = np.nonzero(~bad)[0]
    S, z = pair.gpu_state()
    assert_parity(S[good], pair.S[good], torch.bfloat16, "state S", units="state")
    assert_parity(z[good], pair.z[good], torch.bfloat16, "state z", units="state")
    skipped = torch.as_tensor(np.nonzero(bad)[0], device="cuda")
    assert torch.equal(pair.pool.slab.view(n, -1)[skipped], before[skipped])
