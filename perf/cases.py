"""The work this library is used for, as cases that can be timed and compared.

A case names a kind of call (``op``), the attention configuration and the batch:

  step         one denoising step, hybrid_block_attn
  step_commit  one denoising step with the commit of its block, hybrid_block_attn_commit
  block        a whole block of a decode loop: ``steps`` denoising steps, each on the
               block's newest Q, K and V, then hybrid_commit_block with the last K and V
  logical      step_commit on states kept in the logical layout,
               hybrid_block_attn_commit_logical
  prefill      prompts of different lengths folded into empty states,
               hybrid_commit_ragged
  feature_map  phi of a batch of rows, hybrid_feature_map
  train        forward and backward of the training form

``B`` is the block size, ``Hq`` / ``Hkv`` the query and state heads, ``d`` the head
size, ``F`` the columns of the feature map's W, ``n`` the requests (train: sequences,
feature_map: rows).  ``prefix`` is the longest committed prefix (tokens) of a batch;
requests hold a quarter of it to all of it.  ``k_scale`` scales the keys.

Inputs follow paper_2608_06628_gb300/workloads.py: Q, K, V ~ N(0, 1) rounded to the
I/O type, W ~ N(0, 1/d), alpha ~ U(0, 1).
"""
import numpy as np
import torch

from paper_2608_06628_gb300 import hybrid as H
from paper_2608_06628_gb300.state_pool import StatePool

DEVICE = "cuda"
DTYPES = {"float32": torch.float32, "bfloat16": torch.bfloat16}
ELEM = {"float32": 4, "bfloat16": 2}


def _case(name, op, dtype, n, Hq, Hkv, d, F, B, prefix=0, k_scale=1.0, steps=0, tokens=0):
    c = {"op": op, "dtype": dtype, "n": n, "Hq": Hq, "Hkv": Hkv, "d": d, "F": F, "B": B, "prefix": prefix,
         "k_scale": k_scale, "steps": steps, "tokens": tokens}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one small request in float32, as a numerical reference run is made: all latency
        _case("step_fp32_single", "step", "float32", 1, 2, 2, 64, 64, 16, 64),
        # the last step of a block for a few users, multi-head: the low-batch serving case
        _case("step_commit_mha_b8", "step_commit", "bfloat16", 8, 16, 16, 128, 128, 32, 2048),
        # one denoising step of a full decode batch, grouped queries, ragged prefixes
        _case("step_gqa_b64", "step", "bfloat16", 64, 16, 4, 128, 128, 32, 2048),
        # the same batch's last step of a block, which also folds the block into the states
        _case("step_commit_gqa_b64", "step_commit", "bfloat16", 64, 16, 4, 128, 128, 32, 2048),
        # one layer's share of a decode loop: eight denoising steps and the commit
        _case("block_mha_b32", "block", "bfloat16", 32, 16, 16, 128, 128, 32, 1024, steps=8),
        # the largest serving state: 256 requests, F 256, blocks of 64, sharp keys
        _case("step_commit_f256_b256", "step_commit", "bfloat16", 256, 16, 16, 128, 256, 64, 1024, k_scale=8.0),
        # blocks of 64 tokens with four query heads to a state head: 256 query rows to a state
        _case("step_commit_gqa_blk64", "step_commit", "bfloat16", 32, 16, 4, 128, 128, 64, 1024),
        # a small batch of a whole layer in float32, as a model is validated before it is served
        _case("step_commit_fp32_b8", "step_commit", "float32", 8, 16, 4, 128, 128, 32, 1024),
        # prompts of 1 to 4096 tokens folded into fresh states before decoding starts
        _case("prefill_ragged_b64", "prefill", "bfloat16", 64, 16, 4, 128, 128, 32, tokens=4096),
        # a host that keeps its own states in the logical layout
        _case("logical_gqa_b16", "logical", "bfloat16", 16, 16, 4, 128, 128, 32, 1024),
        # features of a batch of queries, as the attention maps are inspected or distilled
        _case("feature_map_4k", "feature_map", "bfloat16", 4096, 16, 4, 128, 128, 32),
        # a training batch of attention transfer: gradients of the feature maps and gates
        _case("train_8x1024", "train", "bfloat16", 8, 16, 4, 128, 128, 32, tokens=1024),
    ]


def _log_int(rng, lo, hi):
    return int(round(np.exp(rng.uniform(np.log(lo), np.log(hi)))))


def draw(rng):
    op = rng.choice(["step", "step", "step_commit", "step_commit", "block", "prefill", "logical", "feature_map", "train"])
    dtype = "float32" if op in ("step", "step_commit", "feature_map") and rng.random() < 0.25 else "bfloat16"
    Hq, Hkv = rng.choice([(16, 16), (16, 4), (16, 8), (8, 8), (8, 2), (32, 8)])
    d = rng.choice([128, 128, 64])
    F = rng.choice([128, 128, 64, 256, 32])

    def batch(most, work, per_item):
        """A batch size up to ``most`` whose work stays below a listed case's."""
        return _log_int(rng, 1, max(1, min(most, work // per_item)))

    if op == "feature_map":
        return _case(None, op, dtype, batch(4096, 4096 * 16 * 128, Hq * F), Hq, Hkv, d, F, 32)
    if op == "prefill":
        F = rng.choice([64, 128, 128, 256])
        tokens = _log_int(rng, 16, 4096)
        return _case(None, op, dtype, batch(64, 64 * 4096 * 4 * 128, tokens * Hkv * F), Hq, Hkv, d, F, 32, tokens=tokens)
    if op == "train":
        F, B = rng.choice([64, 128]), rng.choice([16, 32])
        blocks = rng.randint(2, 1024 // B)
        return _case(None, op, dtype, batch(8, 1536, blocks * Hkv), Hq, Hkv, d, F, B, tokens=blocks * B)
    k_scale = rng.choice([1.0, 1.0, 1.0, 8.0])
    prefix = 32 * _log_int(rng, 1, 32)
    if op == "block":
        F, B = max(F, 64), rng.choice([16, 32])
        return _case(None, op, dtype, _log_int(rng, 1, 32), Hq, Hkv, d, F, B, prefix, k_scale, steps=rng.randint(2, 8))
    B = rng.choice([16, 32, 32, 64, 48, 24])
    if op == "logical":
        return _case(None, op, dtype, _log_int(rng, 1, 12), Hq, Hkv, d, F, B, prefix, k_scale)
    rows = B * Hq * max(F, 128)
    if dtype == "float32":
        n = batch(8, 8 * 64 * 16 * 128, rows)
    elif B in (16, 32) and F >= 64:
        n = _log_int(rng, 1, 256 if F * Hkv <= 512 else 64)
    else:
        n = batch(32, 32 * 64 * 16 * 128, rows)
    return _case(None, op, dtype, n, Hq, Hkv, d, F, B, prefix, k_scale)


# ------------------------------------------------------------------------- inputs
def _gen(seed, tag):
    g = torch.Generator(device=DEVICE)
    g.manual_seed((int(seed) * 1000003 + tag) & 0x7FFFFFFFFFFFFFFF)
    return g


def _randn(shape, gen, dtype, scale=1.0):
    x = torch.randn(shape, generator=gen, device=DEVICE, dtype=torch.float32)
    return (x * scale if scale != 1.0 else x).to(dtype)


def _params(c, seed):
    dt = DTYPES[c["dtype"]]
    W = _randn((c["Hkv"], c["d"], c["F"]), _gen(seed, 1), dt, c["d"] ** -0.5)
    alpha = torch.rand((c["Hq"],), generator=_gen(seed, 2), device=DEVICE, dtype=torch.float32)
    return W, alpha


def _qkv(c, seed, step):
    dt, g = DTYPES[c["dtype"]], _gen(seed, 10 + step)
    Q = _randn((c["n"], c["B"], c["Hq"], c["d"]), g, dt)
    K = _randn((c["n"], c["B"], c["Hkv"], c["d"]), g, dt, c["k_scale"])
    V = _randn((c["n"], c["B"], c["Hkv"], c["d"]), g, dt)
    return Q, K, V


def _phi(u):
    """Hedgehog features [softmax(u), softmax(-u)] of u = x W."""
    return torch.cat([torch.softmax(u, -1), torch.softmax(-u, -1)], -1)


def _prefix_state(c, seed):
    """S [n, Hkv, 2F, d] and z [n, Hkv, 2F] (float32) of prefixes of prefix/4 .. prefix
    tokens, folded with plain torch a few requests at a time."""
    n, Hkv, d, F, P = c["n"], c["Hkv"], c["d"], c["F"], c["prefix"]
    W = _params(c, seed)[0].float()
    g = _gen(seed, 3)
    lens = torch.randint(max(1, P // 4), P + 1, (n,), generator=g, device=DEVICE)
    S = torch.empty((n, Hkv, 2 * F, d), device=DEVICE)
    z = torch.empty((n, Hkv, 2 * F), device=DEVICE)
    step = max(1, (1 << 27) // (Hkv * P * 2 * F))
    for r in range(0, n, step):
        m = min(step, n - r)
        K = _randn((m, Hkv, P, d), g, torch.float32, c["k_scale"])
        V = _randn((m, Hkv, P, d), g, torch.float32)
        phi = _phi(K @ W)
        phi *= (torch.arange(P, device=DEVICE)[None, :] < lens[r:r + m, None])[:, None, :, None]
        S[r:r + m] = phi.transpose(-1, -2) @ V
        z[r:r + m] = phi.sum(-2)
    return S, z


def _offsets(c, seed):
    """Prompt lengths 1 .. tokens, one of them the longest."""
    rng = np.random.default_rng(int(seed))
    lens = rng.integers(1, c["tokens"] + 1, size=c["n"])
    lens[rng.integers(c["n"])] = c["tokens"]
    return [0] + [int(x) for x in np.cumsum(lens)]


def _prompt(c, seed, total):
    dt, g = DTYPES[c["dtype"]], _gen(seed, 4)
    K = _randn((total, c["Hkv"], c["d"]), g, dt, c["k_scale"])
    V = _randn((total, c["Hkv"], c["d"]), g, dt)
    return K, V


def _train_batch(c, seed):
    dt, g = DTYPES[c["dtype"]], _gen(seed, 5)
    n, L = c["n"], c["tokens"]
    Q = _randn((n, L, c["Hq"], c["d"]), g, dt)
    K = _randn((n, L, c["Hkv"], c["d"]), g, dt)
    V = _randn((n, L, c["Hkv"], c["d"]), g, dt)
    dO = _randn((n, L, c["Hq"], c["d"]), g, dt)
    return Q, K, V, dO


def prepare(case, seed):
    c = case
    cfg = H.make_cfg(c["d"], c["F"], c["Hq"], c["Hkv"], c["B"], DTYPES[c["dtype"]])
    W, alpha = _params(c, seed)
    s = {"op": c["op"], "cfg": cfg, "W": W, "alpha": alpha, "n": c["n"]}
    if c["op"] == "feature_map":
        s["X"] = _randn((c["n"], c["Hq"], c["d"]), _gen(seed, 6), DTYPES[c["dtype"]])
        s["Hq"] = c["Hq"]
        s["Phi"] = torch.empty((c["n"], c["Hq"], 2 * c["F"]), device=DEVICE)
    elif c["op"] == "train":
        s["L"] = c["tokens"]
        s["Q"], s["K"], s["V"], s["dO"] = _train_batch(c, seed)
        s["O"] = torch.empty_like(s["Q"])
        s["bytes"] = H.hybrid_train_workspace_bytes(cfg, c["n"], c["tokens"])
        s["room"] = torch.empty(s["bytes"] + 1024, dtype=torch.uint8, device=DEVICE)
        s["workspace"] = (s["room"].data_ptr() + 1023) & ~1023
        s["dW"] = torch.empty(W.shape, device=DEVICE)
        s["dalpha"] = torch.empty_like(alpha)
    elif c["op"] == "prefill":
        s["offsets"] = _offsets(c, seed)
        s["K"], s["V"] = _prompt(c, seed, s["offsets"][-1])
        s["pool"] = StatePool(cfg, c["n"], DEVICE)
        s["ptrs"] = s["pool"].all_ptrs()
        H.hybrid_state_init(cfg, s["ptrs"], c["n"])
    else:
        s["qkv"] = [_qkv(c, seed, i) for i in range(max(1, c["steps"]))]
        s["O"] = [torch.empty_like(q) for q, _, _ in s["qkv"]]
        S, z = _prefix_state(c, seed)
        if c["op"] == "logical":
            s["S"], s["z"] = S, z
        else:
            s["pool"] = StatePool(cfg, c["n"], DEVICE)
            s["ptrs"] = s["pool"].all_ptrs()
            H.hybrid_state_pack(cfg, S, z, s["ptrs"], c["n"])
    return s


def run(state):
    s = state
    op, cfg, W, alpha, n = s["op"], s["cfg"], s["W"], s["alpha"], s["n"]
    if op == "step":
        Q, K, V = s["qkv"][0]
        H.hybrid_block_attn(cfg, Q, K, V, W, alpha, s["ptrs"], n, s["O"][0])
        return s["O"][0]
    if op == "step_commit":
        Q, K, V = s["qkv"][0]
        H.hybrid_block_attn_commit(cfg, Q, K, V, W, alpha, s["ptrs"], n, s["O"][0])
        return s["O"][0], s["pool"].slab
    if op == "block":
        for (Q, K, V), O in zip(s["qkv"], s["O"]):
            H.hybrid_block_attn(cfg, Q, K, V, W, alpha, s["ptrs"], n, O)
        H.hybrid_commit_block(cfg, K, V, cfg.block_size, W, s["ptrs"], n)
        return s["O"], s["pool"].slab
    if op == "logical":
        Q, K, V = s["qkv"][0]
        H.hybrid_block_attn_commit_logical(cfg, Q, K, V, W, alpha, s["S"], s["z"], n, s["O"][0])
        return s["O"][0], s["S"], s["z"]
    if op == "prefill":
        H.hybrid_commit_ragged(cfg, s["K"], s["V"], s["offsets"], W, s["ptrs"], n)
        return s["pool"].slab
    if op == "feature_map":
        H.hybrid_feature_map(cfg, s["X"], n, s["Hq"], W, s["Phi"])
        return s["Phi"]
    H.hybrid_train_forward(cfg, s["Q"], s["K"], s["V"], W, alpha, n, s["L"], s["O"], s["workspace"], s["bytes"])
    H.hybrid_train_backward(cfg, s["Q"], s["K"], s["V"], W, alpha, s["dO"], n, s["L"], s["workspace"], s["bytes"],
                            s["dW"], s["dalpha"])
    return s["O"], s["dW"], s["dalpha"]


# ------------------------------------------------------------------------- work
def work(case):
    c = case
    n, Hq, Hkv, d, F, B, es = c["n"], c["Hq"], c["Hkv"], c["d"], c["F"], c["B"], ELEM[c["dtype"]]
    w_bytes = Hkv * d * F * es
    state = n * Hkv * (2 * F * d + 2 * F) * 4

    def step_flops(rows, block):      # U = Q W, phi(Q) S, scores and P V
        return rows * (2 * d * F + 4 * F * d + 4 * block * d)

    def fold_flops(rows):             # U = K W and phi(K)^T V
        return rows * (2 * d * F + 4 * F * d)

    q_rows, k_rows = n * B * Hq, n * B * Hkv
    qo, kv = 2 * q_rows * d * es, 2 * k_rows * d * es
    if c["op"] == "step":
        return {"bytes": qo + kv + state + w_bytes + 4 * Hq, "flops": step_flops(q_rows, B)}
    if c["op"] in ("step_commit", "logical"):
        return {"bytes": qo + kv + 2 * state + w_bytes + 4 * Hq, "flops": step_flops(q_rows, B) + fold_flops(k_rows)}
    if c["op"] == "block":
        # each step waits for the one before it, and needs the states (they fit no cache)
        return {"bytes": c["steps"] * (qo + kv + state + w_bytes) + kv + 2 * state + w_bytes,
                "flops": c["steps"] * step_flops(q_rows, B) + fold_flops(k_rows)}
    if c["op"] == "prefill":
        total = _offsets(c, 0)[-1]    # the lengths' sum differs a little with the seed
        return {"bytes": 2 * total * Hkv * d * es + 2 * state + w_bytes, "flops": fold_flops(total * Hkv)}
    if c["op"] == "feature_map":
        return {"bytes": n * Hq * (d * es + 2 * F * 4) + w_bytes, "flops": 2 * n * Hq * d * F}
    t = n * c["tokens"]
    # forward: O.  Backward: dphi(q) and dR per query row, dphi(k) per key row, dO V^T, dW
    flops = step_flops(t * Hq, B) + fold_flops(t * Hkv)
    flops += t * Hq * (8 * F * d + 2 * B * d + 2 * d * F) + t * Hkv * (4 * F * d + 2 * d * F)
    return {"bytes": t * d * es * (3 * Hq + 2 * Hkv) + w_bytes * 3, "flops": flops}


# ------------------------------------------------------------------------- 64-bit values
def _attn64(Q, K, V, W, alpha, S, z):
    """[n, B, Hq, d] of one step against S [n, Hkv, 2F, d], z [n, Hkv, 2F], all float64."""
    n, B, Hq, d = Q.shape
    G = Hq // K.shape[2]
    q = Q.permute(0, 2, 1, 3)                                      # n Hq B d
    k = K.permute(0, 2, 1, 3).repeat_interleave(G, 1)
    v = V.permute(0, 2, 1, 3).repeat_interleave(G, 1)
    phi = _phi(q @ W.repeat_interleave(G, 0)).reshape(n, -1, G * B, S.shape[2])
    lin_num = (phi @ S).reshape(n, Hq, B, d)
    lin_den = (phi @ z[..., None]).reshape(n, Hq, B, 1)
    s = (q @ k.transpose(-1, -2)) * d ** -0.5
    # numerators and denominators are both scaled by e^-m
    m = s.amax(-1, keepdim=True).clamp_min(0.0)
    e = torch.exp(s - m)
    w = torch.sigmoid(alpha)[None, :, None, None]
    num = w * (e @ v) + lin_num * torch.exp(-m)
    den = w * e.sum(-1, keepdim=True) + lin_den * torch.exp(-m)
    return (num / den).permute(0, 2, 1, 3)


def _fold64(K, V, W, S, z):
    """S, z with the tokens of K, V [n, T, Hkv, d] folded in."""
    phi = _phi(K.permute(0, 2, 1, 3) @ W)
    return S + phi.transpose(-1, -2) @ V.permute(0, 2, 1, 3), z + phi.sum(-2)


def _image(S, z):
    """The documented state buffer (include/hybrid.h) of S [n, Hkv, 2F, d], z, flat."""
    n, Hkv, P2, d = S.shape
    f, e = torch.arange(P2, device=S.device)[:, None], torch.arange(d, device=S.device)[None, :]
    at = (f // 32) * 32 * d + e * 32 + 4 * (((f % 32) // 4) ^ (e % 8)) + f % 4
    out = torch.empty((n, Hkv, P2 * d + P2), dtype=S.dtype, device=S.device)
    out[:, :, at.reshape(-1)] = S.reshape(n, Hkv, -1)
    out[:, :, P2 * d:] = z
    return out.reshape(-1)


def _train64(c, seed):
    Q, K, V, dO = (x.double() for x in _train_batch(c, seed))
    W, alpha = (x.double().requires_grad_(True) for x in _params(c, seed))
    n, L, B, Hkv, G = c["n"], c["tokens"], c["B"], c["Hkv"], c["Hq"] // c["Hkv"]
    nb = L // B

    def blocks(x):                                                  # [n nb, B, H, d]
        return x.reshape(n * nb, B, x.shape[2], x.shape[3])

    phi = _phi(blocks(K).permute(0, 2, 1, 3) @ W)                   # n nb, Hkv, B, 2F
    dS = (phi.transpose(-1, -2) @ blocks(V).permute(0, 2, 1, 3)).reshape(n, nb, Hkv, 2 * c["F"], c["d"])
    dz = phi.sum(-2).reshape(n, nb, Hkv, 2 * c["F"])
    S = (dS.cumsum(1) - dS).reshape(n * nb, Hkv, 2 * c["F"], c["d"])
    z = (dz.cumsum(1) - dz).reshape(n * nb, Hkv, 2 * c["F"])
    O = _attn64(blocks(Q), blocks(K), blocks(V), W, alpha, S, z).reshape(n, L, G * Hkv, c["d"])
    (O * dO).sum().backward()
    return O.detach(), W.grad, alpha.grad


def exact(case, seed):
    c = case
    W, alpha = (x.double() for x in _params(c, seed))
    if c["op"] == "feature_map":
        X = _randn((c["n"], c["Hq"], c["d"]), _gen(seed, 6), DTYPES[c["dtype"]]).double()
        return _phi(torch.einsum("nhd,hdf->nhf", X, W.repeat_interleave(c["Hq"] // c["Hkv"], 0)))
    if c["op"] == "train":
        return _train64(c, seed)
    n, Hkv, P2, d = c["n"], c["Hkv"], 2 * c["F"], c["d"]
    if c["op"] == "prefill":
        offs = _offsets(c, seed)
        K, V = _prompt(c, seed, offs[-1])
        S = torch.zeros((n, Hkv, P2, d), dtype=torch.float64, device=DEVICE)
        z = torch.zeros((n, Hkv, P2), dtype=torch.float64, device=DEVICE)
        for r in range(n):
            a, b = offs[r], offs[r + 1]
            S[r:r + 1], z[r:r + 1] = _fold64(K[None, a:b].double(), V[None, a:b].double(), W, S[r:r + 1], z[r:r + 1])
        return _image(S, z)
    S32, z32 = _prefix_state(c, seed)
    qkv = [_qkv(c, seed, i) for i in range(max(1, c["steps"]))]
    O = [torch.empty(q.shape, dtype=torch.float64, device=DEVICE) for q, _, _ in qkv]
    S, z = S32.double(), z32.double()
    del S32, z32
    for r in range(0, n, 16):           # a few requests at a time
        t = slice(r, r + 16)
        for (Q, K, V), o in zip(qkv, O):
            Kd, Vd = K[t].double(), V[t].double()
            o[t] = _attn64(Q[t].double(), Kd, Vd, W, alpha, S[t], z[t])
        if c["op"] != "step":
            S[t], z[t] = _fold64(Kd, Vd, W, S[t], z[t])
    if c["op"] == "step":
        return O[0]
    if c["op"] == "logical":
        return O[0], S, z
    return (O if c["op"] == "block" else O[0]), _image(S, z)
