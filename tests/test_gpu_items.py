"""CTAs of the split-operand step and of the F = 256 step and commit that walk several items,
unusable state pointers among them (a CTA's first item, its last, neighbours, none), against the
fp64 oracle: every barrier, z buffer and tile slot is used more than twice."""
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


def batch(per_cta, items):
    """Requests (items each) for about per_cta items to an SM, the last round partial."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return int(per_cta * sms) // items + 1


def run(call, wl, bad):
    pair = Pair(wl)
    n = wl.n_req
    pair.build_prefixes(np.where(np.arange(n) % 3 > 0, wl.B, 0))
    ptrs = pair.ptrs.clone()
    ptrs[torch.as_tensor(bad)] = 0
    Q, K, V = wk.block_qkv(wl, "items", pair.dev)
    O = torch.full_like(Q, 7.0)
    before = pair.pool.slab.clone().view(n, -1)
    call(pair.cfg, Q, K, V, pair.W, pair.alpha, ptrs, n, O)
    assert H.hybrid_check(check=False) == (H.HYBRID_ERR_DEVICE if bad.any() else H.HYBRID_OK)
    want = pair.orc.block_attn(h64(Q), h64(K), h64(V), pair.W64, pair.alpha64, pair.S, pair.z)
    good = np.nonzero(~bad)[0]
    assert_parity(h64(O)[good], want[good], BF16, "output", units="out")
    skipped = torch.as_tensor(np.nonzero(bad)[0], device="cuda")
    assert torch.all(O[skipped] == 7.0)
    assert torch.equal(pair.pool.slab.view(n, -1)[skipped], before[skipped])
    return pair, K, V, good


def unusable(n, some):
    r = np.arange(n)
    return (r % 7 == 0) | (r % 11 == 4) | (r % 11 == 5) | (r == n - 1) if some else np.zeros(n, bool)


# (items to a CTA, Hq, Hkv, d, F, B): one item to a unit, two (the last one partial), one tile
# buffer with one state head
@pytest.mark.parametrize("per_cta,Hq,Hkv,d,F,B", [
    (4.3, 4, 4, 64, 32, 24), (3.5, 4, 2, 64, 64, 72), (3.2, 1, 1, 128, 256, 120)])
@pytest.mark.parametrize("some", [False, True])
def test_split_step(per_cta, Hq, Hkv, d, F, B, some):
    n = batch(per_cta, Hkv * -(-Hq // Hkv * B // 128))
    run(H.hybrid_block_attn, wk.Workload("items", BF16, n, Hq, Hkv, d, F, B, 95), unusable(n, some))


@pytest.mark.parametrize("per_cta,Hq,Hkv,d,B", [(4.3, 2, 2, 64, 16), (3.4, 4, 1, 64, 16), (3.2, 2, 2, 128, 32)])
@pytest.mark.parametrize("some", [False, True])
def test_wide_step_commit(per_cta, Hq, Hkv, d, B, some):
    n = batch(per_cta, Hkv)
    pair, K, V, good = run(H.hybrid_block_attn_commit, wk.Workload("items", BF16, n, Hq, Hkv, d, 256, B, 96),
                           unusable(n, some))
    pair.orc.commit(h64(K), h64(V), pair.W64, pair.S, pair.z)
    S, z = pair.gpu_state()
    assert_parity(S[good], pair.S[good], BF16, "state S", units="state")
    assert_parity(z[good], pair.z[good], BF16, "state z", units="state")
