"""The work that a user of this library has it do, as timed cases.

A case is a dict of plain values:

  kind     "forward"  one inference pass of the attention (table prepared beforehand)
           "train"    one training step of the layer: prepare the table from the current feature-map
                      parameters, forward with the state saved, backward with every gradient
           "prefill"  a streaming-form forward whose final state is handed to the decode
           "decode"   one streaming-form step per (sequence, head) from a prefilled state
           "weights"  the attention distributions of the conversion's first stage: the kernel's and the
                      softmax teacher's, for every query row
  B, H, n, d, M       batch, heads, tokens, head size, projections (L = 8 channels of 64 hidden units each)
  io                  "bf16" or "f32"
  causal              streaming form (True) or every key for every query (False)
  min_len             shortest valid length: per-sequence lengths U[min_len, n] (0: no padding)
  ch_rms              target of the channel RMS normalisation (0: off)
  per_head            one feature map per head
  scale               standard deviation of Q, K and V

Inputs are N(0, scale^2) and dO is N(0, 1); the feature-map parameters follow the listing's
initialisation, with a small projection bias as training leaves one.
"""
from __future__ import annotations

import math

import torch

import paper_2512_08061_gb300.luna as luna

L, HIDDEN, EPS = 8, 64, 1e-6
DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


def _case(name, kind, B, H, n, d, M, io="bf16", causal=False, min_len=0, ch_rms=0.0, per_head=False, scale=1.0):
    c = dict(kind=kind, B=B, H=H, n=n, d=d, M=M, io=io, causal=causal, min_len=min_len, ch_rms=ch_rms,
             per_head=per_head, scale=scale)
    return {"name": name, **c} if name else c


def listed():
    s32, s64, s128 = 1 / math.sqrt(32), 1 / math.sqrt(64), 1 / math.sqrt(128)
    return [
        # the smallest call: one head of 256 tokens in fp32, where launches and latency are everything
        _case("tiny_f32_forward", "forward", 1, 1, 256, 64, 8, "f32"),
        # ViT-B/16 inference: many short, ragged (197-token) sequences
        _case("vit_forward", "forward", 64, 12, 197, 64, 8),
        # BERT-base fine-tuning step of one layer
        _case("bert_train", "train", 32, 12, 512, 64, 8),
        # Long Range Arena encoder trained from scratch, padded batches
        _case("lra_train", "train", 32, 4, 4096, 32, 8, min_len=2048, scale=s32),
        # the same with the listing's channel RMS normalisation
        _case("lra_train_ch_rms", "train", 32, 4, 4096, 32, 8, min_len=2048, ch_rms=0.05, scale=s32),
        # long-context streaming form, the largest training step
        _case("causal_long_train", "train", 2, 32, 65536, 128, 16, causal=True, scale=s128),
        # serving: the prefill of 64 sequences, whose state the decode continues
        _case("prefill", "prefill", 64, 32, 1024, 128, 16, causal=True, scale=s128),
        # serving: one token for each of 64 sequences
        _case("decode", "decode", 64, 32, 1024, 128, 16, causal=True, scale=s128),
        # serving: one token of a single sequence, pure latency
        _case("decode_single", "decode", 1, 12, 200, 64, 8, causal=True, scale=s64),
        # fp32 training (the precision the listing runs in) at the BERT-base layer shape
        _case("bert_train_f32", "train", 8, 12, 512, 64, 8, "f32"),
        # streaming-form training at the common head size of 64
        _case("causal_train_d64", "train", 8, 12, 1024, 64, 8, causal=True, scale=s64),
        # conversion, stage 1: both attention distributions of one BERT-base layer
        _case("conversion_weights", "weights", 4, 12, 512, 64, 8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("forward", "train", "train", "train", "prefill", "decode", "weights"))
    causal = kind in ("prefill", "decode") or (kind != "weights" and rng.random() < 0.4)
    io = rng.choice(("bf16", "bf16", "f32"))
    d, M = rng.choice(((32, 8), (64, 8), (64, 8), (128, 16), (128, 16), (48, 8), (96, 8), (64, 16)))
    H = rng.choice((1, 2, 3, 4, 8, 12, 16, 32))
    n = _log_int(rng, 16, 1024) if kind == "weights" else _log_int(rng, 16, 1500) if kind == "decode" else \
        _log_int(rng, 16, 65536)
    # rows of one pass: bounded by what the listed cases of the same kind and arithmetic hold
    fast = io == "bf16" and (d, M) in (((128, 16),) if causal else ((32, 8), (64, 8)))
    rows = {"decode": 64 * 32 * 1024, "weights": 4 * 12 * 512 * 512 // n}.get(kind, (1 << 21) if fast else 100_000)
    rows = max(rows * 64 // (d if fast or kind in ("decode", "weights") else max(d, M * L)), n)
    H = max(1, min(H, rows // n))
    B = _log_int(rng, 1, max(1, min(64, rows // (n * H))))
    pad = kind in ("forward", "train") and n >= 32 and rng.random() < 0.4
    ch_rms = 0.05 if kind == "train" and rng.random() < 0.1 else 0.0
    per_head = kind in ("forward", "train") and not ch_rms and H <= 12 and rng.random() < 0.15
    scale = rng.choice((1.0, 1 / math.sqrt(d)))
    return _case("", kind, B, H, n, d, M, io, causal, n // 2 if pad else 0, ch_rms, per_head, scale)


# ---------------------------------------------------------------------------
# inputs

def _randn(g, shape, scale, dtype):
    out = torch.empty(shape, dtype=dtype, device="cuda")
    return out.normal_(0.0, scale, generator=g)


def _params(c, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 2 + 1)
    sets = (c["H"],) if c["per_head"] else ()
    d, M, f = c["d"], c["M"], dict(device="cuda", dtype=torch.float32)

    def uniform(shape, bound):
        return torch.empty(sets + shape, **f).uniform_(-bound, bound, generator=g)

    return {"W": torch.empty(sets + (M, d), **f).normal_(0.0, 1 / math.sqrt(d), generator=g),
            "b": torch.empty(sets + (M,), **f).normal_(0.0, 0.1, generator=g),
            "w1": uniform((L, HIDDEN), 1.0), "b1": uniform((L, HIDDEN), 1.0),
            "w2": uniform((L, HIDDEN), 1 / math.sqrt(HIDDEN)), "b2": uniform((L,), 1 / math.sqrt(HIDDEN))}


def _inputs(c, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 2)
    shape, dt = (c["B"], c["H"], c["n"], c["d"]), DTYPES[c["io"]]
    x = {"Q": _randn(g, shape, c["scale"], dt), "K": _randn(g, shape, c["scale"], dt), "lengths": None}
    if c["kind"] != "weights":
        x["V"] = _randn(g, shape, c["scale"], dt)
    if c["kind"] == "train":
        x["dO"] = _randn(g, shape, 1.0, dt)
    if c["min_len"]:
        x["lengths"] = torch.randint(c["min_len"], c["n"] + 1, (c["B"],), generator=g, device="cuda", dtype=torch.int32)
    if c["kind"] == "decode":
        one = (c["B"], c["H"], c["d"])
        x.update({k: _randn(g, one, c["scale"], dt) for k in ("q", "k", "v")})
    return x


def _state_views(lu, c):
    """The final S and z of a streaming-form layer as views of its state buffer."""
    S, Ss, z, zs = luna.luna_state_final(lu.ad, lu.pd, lu.state)
    flat, D, d = lu.state.view(torch.float32), c["M"] * L, c["d"]
    at = [(p - lu.state.data_ptr()) // 4 for p in (S, z)]
    BH = (c["B"], c["H"])
    return (torch.as_strided(flat, BH + (D, d), (c["H"] * Ss, Ss, d, 1), at[0]),
            torch.as_strided(flat, BH + (D,), (c["H"] * zs, zs, 1), at[1]))


def prepare(case, seed):
    c, x, p = case, _inputs(case, seed), _params(case, seed)
    s = {"kind": c["kind"], "x": x, "params": p, "case": c}
    if c["kind"] == "weights":
        s["pd"] = luna.phi_desc(c["M"], L, HIDDEN)
        s["ad"] = luna.attn_desc(c["B"], c["H"], c["n"], c["d"], c["d"], False, 0, EPS, luna._DTYPES[DTYPES[c["io"]]])
        s["table"] = luna.alloc_bytes(luna.luna_phi_table_size(s["pd"], c["d"]), "cuda")
        luna.luna_phi_prepare(s["pd"], c["d"], p, s["table"])
        return s
    lu = s["layer"] = luna.Luna(c["B"], c["H"], c["n"], c["d"], c["d"], c["M"], L, HIDDEN, c["causal"], EPS,
                                DTYPES[c["io"]], ch_rms_target=c["ch_rms"], per_head=c["per_head"])
    if c["kind"] != "train":
        lu.prepare(p)
    if c["kind"] in ("prefill", "decode"):
        s["state"] = _state_views(lu, c)
    if c["kind"] == "decode":
        lu.forward(x.pop("Q"), x.pop("K"), x.pop("V"))
    return s


def run(state):
    x = state["x"]
    if state["kind"] == "weights":
        c = state["case"]
        A, P = (torch.empty((c["B"], c["H"], c["n"], c["n"]), dtype=torch.float32, device="cuda") for _ in range(2))
        for out, teacher in ((A, False), (P, True)):
            luna.luna_attn_weights(state["ad"], state["pd"], state["table"], x["Q"], x["K"], None, 0, c["n"], teacher, out)
        return {"student": A, "teacher": P}
    lu = state["layer"]
    if state["kind"] == "decode":
        o = lu.decode(x["q"], x["k"], x["v"])
        return {"o": o, "S": state["state"][0], "z": state["state"][1]}
    if state["kind"] == "train":
        lu.prepare(state["params"])
        O = lu.forward(x["Q"], x["K"], x["V"], x["lengths"])
        return {"O": O, **lu.backward(x["Q"], x["K"], x["V"], x["dO"], x["lengths"])}
    if state["kind"] == "prefill":
        O = lu.forward(x["Q"], x["K"], x["V"], x["lengths"])
        return {"O": O, "S": state["state"][0], "z": state["state"][1]}
    return {"O": lu.forward(x["Q"], x["K"], x["V"], x["lengths"], save_state=False)}


def work(case):
    c = case
    eb, d, M, D = (2 if c["io"] == "bf16" else 4), c["d"], c["M"], c["M"] * L
    heads = c["B"] * c["H"]
    R = heads * c["n"]
    Rv = R * (1 + c["min_len"] / c["n"]) / 2 if c["min_len"] else R  # valid rows, on average
    par = 4 * (M * d + M + 3 * L * HIDDEN + L) * (c["H"] if c["per_head"] else 1)
    stat = 4 * heads * (D * d + D)
    fwd = 4 * M * d + 4 * D * d + 4 * D
    if c["kind"] == "decode":
        return {"bytes": 2 * stat + heads * 4 * d * eb + par, "flops": heads * fwd}
    if c["kind"] == "weights":
        pairs = heads * c["n"] ** 2
        return {"bytes": 2 * R * d * eb + 8 * pairs + par, "flops": 4 * M * d * R + pairs * (2 * D + 2 * d)}
    if c["kind"] == "train":
        return {"bytes": Rv * 4 * d * eb + R * 4 * d * eb + 2 * par, "flops": Rv * (fwd + 12 * M * d + 10 * D * d + 6 * D)}
    return {"bytes": Rv * 3 * d * eb + R * d * eb + par + (stat if c["kind"] == "prefill" else 0), "flops": Rv * fwd}


# ---------------------------------------------------------------------------
# the same in 64 bits with plain torch: every hidden unit, every projection, autograd through the channel
# MLPs, the attention and its gradient from their definitions

_CHUNK = 128  # rows per chunk of the streaming form


def _bank(x, p):
    """The channel MLPs' outputs (rows, M, L) of rows x."""
    u = x @ p["W"].T + p["b"]
    h = torch.relu(torch.addcmul(p["b1"], u[:, :, None, None], p["w1"]))
    return torch.relu((h * p["w2"]).sum(-1) + p["b2"])


def _row_chunks(rows, M):
    step = max(1, (1 << 27) // (M * L * HIDDEN))
    return [(i, min(rows, i + step)) for i in range(0, rows, step)]


def _bank_all(X, p):
    """(..., n, d) in the I/O type -> (..., n, M, L) in 64 bits."""
    flat, M = X.reshape(-1, X.shape[-1]), p["W"].shape[0]
    out = torch.empty((flat.shape[0], M, L), dtype=torch.float64, device=X.device)
    for a, b in _row_chunks(flat.shape[0], M):
        out[a:b] = _bank(flat[a:b].double(), p)
    return out.reshape(X.shape[:-1] + (M, L))


def _bank_backward(X, dy, p, grads):
    """dX of the channel MLPs; adds the parameter gradients to grads."""
    flat, dflat, M = X.reshape(-1, X.shape[-1]), dy.reshape(-1, *dy.shape[-2:]), p["W"].shape[0]
    dX = torch.empty(flat.shape, dtype=torch.float64, device=X.device)
    keys = list(p)
    for a, b in _row_chunks(flat.shape[0], 4 * M):
        x = flat[a:b].double().requires_grad_()
        q = {k: v.detach().requires_grad_() for k, v in p.items()}
        with torch.enable_grad():
            y = _bank(x, q)
        got = torch.autograd.grad(y, [x] + [q[k] for k in keys], dflat[a:b])
        dX[a:b] = got[0]
        for k, v in zip(keys, got[1:]):
            grads["d" + k] += v
    return dX.reshape(X.shape)


def _chunks(t):
    n = t.shape[-2]
    pad = -n % _CHUNK
    t = torch.nn.functional.pad(t, (0, 0, 0, pad)) if pad else t
    return t.reshape(t.shape[:-2] + (-1, _CHUNK, t.shape[-1]))


def _rows(t, n):
    return t.reshape(t.shape[:-3] + (-1, t.shape[-1]))[..., :n, :]


def _attend(pq, pk, V1, causal):
    """phi(Q) (phi(K)^T [V, 1]) over every key, or over the keys up to each row; and the final statistics."""
    if not causal:
        S = pk.transpose(-1, -2) @ V1
        return pq @ S, S
    n = pq.shape[-2]
    q, k, v = _chunks(pq), _chunks(pk), _chunks(V1)
    part = k.transpose(-1, -2) @ v
    run = part.cumsum(-3)
    num = q @ (run - part) + torch.tril(q @ k.transpose(-1, -2)) @ v
    return _rows(num, n), run[..., -1, :, :]


def _attend_backward(pq, pk, V1, G, causal):
    """Gradients of _attend's product for its gradient G: phi(Q), phi(K), V."""
    if not causal:
        S, T = pk.transpose(-1, -2) @ V1, pq.transpose(-1, -2) @ G
        return G @ S.transpose(-1, -2), V1 @ T.transpose(-1, -2), pk @ T
    n = pq.shape[-2]
    q, k, v, g = _chunks(pq), _chunks(pk), _chunks(V1), _chunks(G)
    part = k.transpose(-1, -2) @ v
    before = part.cumsum(-3) - part
    part = q.transpose(-1, -2) @ g
    after = part.flip(-3).cumsum(-3).flip(-3) - part
    C, E = torch.tril(q @ k.transpose(-1, -2)), torch.tril(g @ v.transpose(-1, -2))
    dq = g @ before.transpose(-1, -2) + E @ k
    dk = v @ after.transpose(-1, -2) + E.transpose(-1, -2) @ q
    dv = k @ after + C.transpose(-1, -2) @ g
    return _rows(dq, n), _rows(dk, n), _rows(dv, n)


def _with_ones(V):
    return torch.cat((V.double(), torch.ones(V.shape[:-1] + (1,), dtype=torch.float64, device=V.device)), -1)


def _exact_layer(c, x, p, heads):
    """Outputs of one forward (and backward) of the given heads, whose feature map is p."""
    Q, K, V = (x[k][:, heads] for k in ("Q", "K", "V"))
    B, H, n, d = Q.shape
    M, causal, lengths = c["M"], c["causal"], x["lengths"]
    ln = torch.full((B,), n, device="cuda") if lengths is None else lengths.long()
    mask = (torch.arange(n, device="cuda") < ln[:, None]).double()[:, None, :, None, None]
    count = float(ln.sum()) * H * M
    y, s, rms = {}, {}, {}
    for k, X in (("Q", Q), ("K", K)):
        y[k] = _bank_all(X, p) * mask
        s[k] = torch.ones(L, dtype=torch.float64, device="cuda")
        if c["ch_rms"]:
            rms[k] = y[k].square().sum((0, 1, 2, 3)).div(count).sqrt()
            s[k] = torch.clamp(c["ch_rms"] / (rms[k] + 1e-6), max=1.0)
    phi = {k: (y[k] * s[k]).div_(math.sqrt(M)).reshape(B, H, n, M * L) for k in y}
    O, S = torch.empty((B, H, n, d), dtype=torch.float64, device="cuda"), []
    train = c["kind"] == "train"
    dphi, dV = {k: torch.empty_like(phi[k]) for k in phi} if train else None, torch.empty_like(O) if train else None
    for b in range(B):
        V1 = _with_ones(V[b])
        num, fin = _attend(phi["Q"][b], phi["K"][b], V1, causal)
        den = num[..., d:] + EPS
        ok = (den != 0) & (mask[b, :, :, 0] > 0)
        inv = torch.where(ok, 1.0 / den, torch.zeros_like(den))
        O[b] = num[..., :d] * inv
        S.append(fin)
        if train:
            g = x["dO"][b, heads].double() * inv
            G = torch.cat((g, -(x["dO"][b, heads].double() * O[b]).sum(-1, keepdim=True) * inv), -1)
            dphi["Q"][b], dphi["K"][b], t = _attend_backward(phi["Q"][b], phi["K"][b], V1, G, causal)
            dV[b] = t[..., :d] * mask[b, :, :, 0]
    out = {"O": O}
    if c["kind"] == "prefill":
        S = torch.stack(S)
        out.update(S=S[..., :d], z=S[..., d])
    if train:
        del phi
        out["dV"] = dV
        grads = {"d" + k: torch.zeros_like(v) for k, v in p.items()}
        for k, X in (("Q", Q), ("K", K)):
            dy = dphi.pop(k).reshape(B, H, n, M, L).div_(math.sqrt(M)).mul_(mask)
            if c["ch_rms"]:
                ds = (dy * y[k]).sum((0, 1, 2, 3))
                r = rms[k]
                dr = torch.where(c["ch_rms"] / (r + 1e-6) <= 1, -ds * c["ch_rms"] / (r + 1e-6) ** 2, torch.zeros_like(r))
                dy = dy * s[k] + y[k] * (dr / (count * r))
            out["d" + k] = _bank_backward(X, dy, p, grads) * mask[..., 0]
        out.update(grads)
    return out


@torch.no_grad()
def exact(case, seed):
    c, x = case, _inputs(case, seed)
    p = {k: v.double() for k, v in _params(case, seed).items()}
    if c["kind"] == "weights":
        pq, pk = (_bank_all(x[k], p).reshape(c["B"], c["H"], c["n"], -1) / math.sqrt(c["M"]) for k in ("Q", "K"))
        k = pq @ pk.transpose(-1, -2)
        t = x["Q"].double() @ x["K"].double().transpose(-1, -2) / math.sqrt(c["d"])
        return {"student": k / (k.sum(-1, keepdim=True) + EPS), "teacher": torch.softmax(t, -1)}
    if c["kind"] == "decode":
        pk, kn, qn = (_bank_all(v, p).flatten(-2) / math.sqrt(c["M"]) for v in (x["K"], x["k"], x["q"]))
        S = pk.transpose(-1, -2) @ _with_ones(x["V"]) + kn[..., None] * _with_ones(x["v"])[..., None, :]
        num = (qn[..., None, :] @ S)[..., 0, :]
        return {"o": num[..., :-1] / (num[..., -1:] + EPS), "S": S[..., :-1], "z": S[..., -1]}
    if not c["per_head"]:
        return _exact_layer(c, x, p, slice(None))
    per = [_exact_layer(c, x, {k: v[h] for k, v in p.items()}, slice(h, h + 1)) for h in range(c["H"])]
    shared = ("O", "dQ", "dK", "dV")
    return {k: torch.cat([o[k] for o in per], 1) if k in shared else torch.stack([o[k] for o in per]) for k in per[0]}
