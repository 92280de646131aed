"""Pack and unpack of the state image for every tile count and head size, logical buffers
that are only 4-byte aligned, and a bad pointer in the batch: the documented offsets, and
nothing outside the buffers written."""
import pytest
import torch

from paper_2608_06628_gb300 import hybrid as H
from paper_2608_06628_gb300.state_pool import StatePool

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("d,F", [(64, 16), (128, 16), (64, 32), (128, 64), (64, 128), (128, 256)])
def test_pack_unpack(d, F, off):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n, Hkv, P2 = 5, 3, 2 * F
    cfg = H.make_cfg(d, F, 3, Hkv, 16, torch.bfloat16)
    pool = StatePool(cfg, n, "cuda")
    pool.slab.fill_(7.0)
    g = torch.Generator(device="cuda").manual_seed(d + F + off)

    def flat(numel):   # a buffer with guard values around numel floats, off floats past alignment
        b = torch.full((numel + 8,), 9.0, device="cuda")
        return b, b[off:off + numel]

    Sb, S = flat(n * Hkv * P2 * d)
    zb, z = flat(n * Hkv * P2)
    S.copy_(torch.randn(S.shape, generator=g, device="cuda"))
    z.copy_(torch.randn(z.shape, generator=g, device="cuda"))
    ptrs = pool.all_ptrs()
    ptrs[1] = 0                      # request 1: reported and skipped
    H.hybrid_state_pack(cfg, S, z, ptrs, n)
    assert H.hybrid_check(check=False) == H.HYBRID_ERR_DEVICE
    f, e = torch.arange(P2, device="cuda")[:, None], torch.arange(d, device="cuda")[None, :]
    at = ((f // 32) * 32 * d + e * 32 + 4 * (((f % 32) // 4) ^ (e % 8)) + f % 4).reshape(-1)
    want = torch.empty((n, Hkv, P2 * d + P2), device="cuda")
    want[:, :, at] = S.view(n, Hkv, -1)
    want[:, :, P2 * d:] = z.view(n, Hkv, -1)
    want[1] = 7.0
    assert torch.equal(pool.slab.view(n, Hkv, -1), want)
    S2b, S2 = flat(S.numel())
    z2b, z2 = flat(z.numel())
    H.hybrid_state_unpack(cfg, ptrs, n, S2, z2)
    assert H.hybrid_check(check=False) == H.HYBRID_ERR_DEVICE
    keep = [i for i in range(n) if i != 1]
    assert torch.equal(S2.view(n, -1)[keep], S.view(n, -1)[keep]) and torch.all(S2.view(n, -1)[1] == 9.0)
    assert torch.equal(z2.view(n, -1)[keep], z.view(n, -1)[keep]) and torch.all(z2.view(n, -1)[1] == 9.0)
    for b in (S2b, z2b):
        assert torch.all(b[:off] == 9.0) and torch.all(b[off - 8:] == 9.0)
