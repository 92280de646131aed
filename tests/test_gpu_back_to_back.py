"""Steps and commits issued one behind the other, so that a kernel starts while the one in front
still writes the states: the same bits as with the device idle between the calls."""
import pytest
import torch

from gpu_harness import Pair
from paper_2608_06628_gb300 import hybrid as H
from paper_2608_06628_gb300 import workloads as wk

pytestmark = pytest.mark.gpu

BF16, F32 = torch.bfloat16, torch.float32


@pytest.mark.parametrize("dt,n,Hq,Hkv,d,F,B", [
    (F32, 1, 2, 2, 64, 64, 16), (F32, 8, 16, 4, 128, 128, 32), (F32, 40, 4, 2, 64, 256, 24), (BF16, 2, 6, 2, 128, 128, 48),
    (BF16, 4, 16, 4, 128, 128, 64), (BF16, 20, 8, 8, 64, 32, 24), (BF16, 6, 8, 4, 128, 256, 40)])
def test_same_bits(dt, n, Hq, Hkv, d, F, B):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_06628_gb300 import build
    build.build()
    wl = wk.Workload("chain", dt, n, Hq, Hkv, d, F, B, 97)
    blocks = [wk.block_qkv(wl, i, "cuda") for i in range(12)]

    def run(wait):
        pair = Pair(wl, tracked=[0])
        O = [torch.empty_like(Q) for Q, _, _ in blocks for _ in range(2)]
        torch.cuda.synchronize()
        for i, (Q, K, V) in enumerate(blocks):
            H.hybrid_block_attn(pair.cfg, Q, K, V, pair.W, pair.alpha, pair.ptrs, n, O[2 * i])
            wait()
            H.hybrid_block_attn_commit(pair.cfg, Q, K, V, pair.W, pair.alpha, pair.ptrs, n, O[2 * i + 1])
            wait()
        H.hybrid_check()
        return O + [pair.pool.slab.clone()]

    want = run(torch.cuda.synchronize)
    for _ in range(3):
        assert all(torch.equal(a, b) for a, b in zip(run(lambda: None), want))
