"""Infinities and NaN in V and in the state: an output element is what float64 gives, infinite
with the same sign or NaN, and the elements beside it stay what they are without them."""
import numpy as np
import pytest
import torch

from gpu_harness import assert_parity, h64, Pair
from paper_2608_06628_gb300 import hybrid as H
from paper_2608_06628_gb300 import workloads as wk

pytestmark = pytest.mark.gpu

BF16, F32 = torch.bfloat16, torch.float32
INF, NAN = float("inf"), float("nan")


def agree(got, want, dt, what, units):
    """Infinities and NaN in the same places, the rest within the bound of the type."""
    for kind in (np.isposinf, np.isneginf, np.isnan):
        assert np.array_equal(kind(got), kind(want)), f"{what}: {kind.__name__} differs"
    fin = np.isfinite(want)
    assert_parity(np.where(fin, got, 0.0), np.where(fin, want, 0.0), dt, what, units=units)


# (dtype, n, Hq, Hkv, d, F, B): the split-operand step, its F = 256 form, one state tile; step
# and commit at F = 256; the streaming kernels; the CUDA cores
@pytest.mark.parametrize("dt,n,Hq,Hkv,d,F,B", [
    (BF16, 2, 4, 1, 128, 128, 64), (BF16, 3, 2, 2, 128, 64, 24), (BF16, 2, 8, 1, 64, 256, 40), (BF16, 2, 2, 2, 64, 16, 20),
    (BF16, 2, 2, 2, 128, 256, 64), (BF16, 3, 8, 2, 64, 256, 16), (BF16, 3, 4, 1, 128, 128, 32), (BF16, 2, 2, 2, 64, 64, 16),
    (BF16, 2, 2, 1, 128, 128, 48),
    (F32, 2, 4, 2, 64, 64, 17), (BF16, 2, 6, 2, 128, 128, 48),
])
@pytest.mark.parametrize("where", ["values", "state"])
def test_step_commit(dt, n, Hq, Hkv, d, F, B, where):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_06628_gb300 import build
    build.build()
    wl = wk.Workload("nonfinite", dt, n, Hq, Hkv, d, F, B, 92)
    pair = Pair(wl)
    pair.build_prefixes(np.full(n, 2 * B))
    Q, K, V = wk.block_qkv(wl, "nonfinite", pair.dev)
    if where == "values":
        V[0, 3, 0, 5] = INF
        V[0, B - 1, 0, 9] = -INF
        V[0, 0, 0, 17], V[0, 2, 0, 17] = INF, -INF
        V[n - 1, 1, Hkv - 1, 30] = NAN
    else:
        S = torch.as_tensor(pair.S, dtype=F32, device=pair.dev).contiguous()
        z = torch.as_tensor(pair.z, dtype=F32, device=pair.dev).contiguous()
        S[0, 0, 3, 5] = INF
        S[0, 0, 2 * F - 1, 9] = -INF
        S[0, 0, 1, 17], S[0, 0, F + 2, 17] = INF, -INF
        S[n - 1, Hkv - 1, F, 30] = NAN
        H.hybrid_state_pack(pair.cfg, S, z, pair.ptrs, n)
        pair.S, pair.z = h64(S), h64(z)
    want = pair.orc.block_attn(h64(Q), h64(K), h64(V), pair.W64, pair.alpha64, pair.S, pair.z)
    pair.orc.commit(h64(K), h64(V), pair.W64, pair.S, pair.z)
    O = torch.empty_like(Q)
    H.hybrid_block_attn_commit(pair.cfg, Q, K, V, pair.W, pair.alpha, pair.ptrs, n, O)
    H.hybrid_check()
    assert np.isinf(want).any() and np.isnan(want).any()
    agree(h64(O), want, dt, "output", "out")
    S, z = pair.gpu_state()
    agree(S, pair.S, dt, "state S", "state")
    assert_parity(z, pair.z, dt, "state z", units="state")
