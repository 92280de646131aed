"""The state of a short commit is the same bits from whichever kernel folds it, and the bits of
a one-chunk prompt are the same from run to run."""
import pytest
import torch

from gpu_harness import Pair
from paper_2608_06628_gb300 import hybrid as H
from paper_2608_06628_gb300 import workloads as wk

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_06628_gb300 import build
    build.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("T", [32, 21, 5])
def test_batch_size_does_not_change_a_state(T):
    """d = F = 128, up to 32 tokens: half a wave of units, one to three waves, more than three."""
    Hkv, sms = 4, torch.cuda.get_device_properties(0).multi_processor_count
    sizes = [sms // (2 * Hkv), sms // (2 * Hkv) + 1, 2 * sms // Hkv, 3 * sms // Hkv + 1]
    wl = wk.Workload("batch", torch.bfloat16, sizes[-1], Hkv, Hkv, 128, 128, 32, 93)
    K0, V0 = wk.prefix_kv(wl, 0, "cuda", n_tok=40)
    K, V = wk.prefix_kv(wl, 1, "cuda", n_tok=T)
    slabs = []
    for n in sizes:
        pair = Pair(wl, tracked=[0])
        H.hybrid_commit_block(pair.cfg, K0, V0, 40, pair.W, pair.ptrs, wl.n_req)
        for r in range(0, wl.n_req, n):
            m = min(n, wl.n_req - r)
            # (a last, smaller batch is folded in any case: another side of the rule)
            H.hybrid_commit_block(pair.cfg, K[r:r + m], V[r:r + m], T, pair.W, pair.ptrs[r:r + m], m)
        H.hybrid_check()
        slabs.append(pair.pool.slab.clone())
    for s in slabs[1:]:
        assert torch.equal(s, slabs[0])


@pytest.mark.parametrize("d,F", [(128, 128), (64, 128), (128, 64), (64, 64)])
def test_one_chunk_prompt_repeats_bitwise(d, F):
    """65 to 128 tokens per request (four warps' token sums): the same bits from run to run."""
    wl = wk.Workload("repeat", torch.bfloat16, 400, 2, 2, d, F, 32, 94)
    K, V = wk.prefix_kv(wl, 75, "cuda", n_tok=128)
    slabs = []
    for _ in range(6):
        pair = Pair(wl, tracked=[0])
        for T in (128, 100, 70):
            H.hybrid_commit_block(pair.cfg, K[:, :T].contiguous(), V[:, :T].contiguous(), T, pair.W, pair.ptrs, wl.n_req)
        H.hybrid_check()
        slabs.append(pair.pool.slab.clone())
    assert all(torch.equal(s, slabs[0]) for s in slabs)
