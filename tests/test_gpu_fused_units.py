"""Fused step and commit over CTAs of several units, with unusable state pointers among them
(a CTA's first unit, its last one, both, none): the others' outputs and states against the
fp64 oracle, nothing written for the skipped requests."""
import numpy as np
import pytest
import torch

from gpu_harness import Pair, assert_parity, h64
from paper_2608_06628_gb300 import hybrid as H
from paper_2608_06628_gb300 import workloads as wk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,Hq,Hkv,d,F", [(320, 2, 1, 64, 64), (480, 1, 1, 128, 128), (330, 4, 1, 64, 128)])
def test_skipped_units(n, Hq, Hkv, d, F):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_06628_gb300 import build
    build.build()
    wl = wk.Workload("units", torch.bfloat16, n, Hq, Hkv, d, F, 32, 65)
    pair = Pair(wl)
    pair.build_prefixes(np.arange(n) % 2 * 32)
    bad = np.array([r % 7 in (0, 3) or r % 11 in (4, 5) or r == n - 1 for r in range(n)])
    ptrs = pair.ptrs.clone()
    ptrs[torch.as_tensor(bad)] = 0
    before = pair.pool.slab.clone().view(n, -1)
    Q, K, V = wk.block_qkv(wl, "units", pair.dev)
    O = torch.full_like(Q, 7.0)
    H.hybrid_block_attn_commit(pair.cfg, Q, K, V, pair.W, pair.alpha, ptrs, n, O)
    assert H.hybrid_check(check=False) == H.HYBRID_ERR_DEVICE
    want = pair.orc.block_attn(h64(Q), h64(K), h64(V), pair.W64, pair.alpha64, pair.S, pair.z)
    pair.orc.commit(h64(K), h64(V), pair.W64, pair.S, pair.z)
    good = np.nonzero(~bad)[0]
    assert_parity(h64(O)[good], want[good], torch.bfloat16, "output", units="out")
    S, z = pair.gpu_state()
    assert_parity(S[good], pair.S[good], torch.bfloat16, "state S", units="state")
    assert_parity(z[good], pair.z[good], torch.bfloat16, "state z", units="state")
    skipped = torch.as_tensor(np.nonzero(bad)[0], device="cuda")
    assert torch.all(O[skipped] == 7.0)
    assert torch.equal(pair.pool.slab.view(n, -1)[skipped], before[skipped])
