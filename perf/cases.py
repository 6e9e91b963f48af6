"""The calls this library is timed and checked on: CCQ attention through its public entry points.

Every case is one user-level call (or, for training, the forward and backward calls of one step) of
``paper_2606_01294_gb300.ccq`` on inputs resident on the GPU: token-by-token decoding, prefill of one or
many sequences (fixed length, ragged and resumed, packed), training steps, and the fp32 path, for both
backbones (GLA and Gated DeltaNet).  Sizes are those of the repository's workloads (heads of 128 as in a
2048-wide layer of 16 heads, T = 4096 and 20480, decode batch 256, the fp32 case of two heads of 64) and of
its tests, and the ranges around them.
"""
import math
import random

import torch
import torch.nn.functional as F

from paper_2606_01294_gb300 import ccq

GLA, GDN = ccq.GLA, ccq.GDN
CHUNK = 64


def listed():
    return [
        # One token for a couple of interactive sessions: the smallest call there is, latency and launches.
        dict(name="decode_gla_b2", kind="decode", backbone="gla", B=2, H=16, d=128),
        # One token for a full serving batch: the whole fp32 cache is read and written.
        dict(name="decode_gdn_b256", kind="decode", backbone="gdn", B=256, H=16, d=128),
        # A new turn of one conversation, appended to its cached state: short, ragged, resumed.
        dict(name="prefill_gla_turn", kind="prefill", backbone="gla", B=1, T=1000, H=16, resumed=True),
        dict(name="prefill_gdn_turn", kind="prefill", backbone="gdn", B=2, T=777, H=16, resumed=True),
        # Prefill of a batch of 4K prompts (the headline workload) on each backbone.
        dict(name="prefill_gla_4k", kind="prefill", backbone="gla", B=8, T=4096, H=16, resumed=False),
        dict(name="prefill_gdn_4k", kind="prefill", backbone="gdn", B=8, T=4096, H=16, resumed=False),
        # One long document (length extrapolation): few sequences, many chunks.
        dict(name="prefill_gla_20k", kind="prefill", backbone="gla", B=1, T=20480, H=16, resumed=False),
        dict(name="prefill_gdn_20k", kind="prefill", backbone="gdn", B=1, T=20480, H=16, resumed=False),
        # A serving mix: 64 prompts of very different lengths packed into one call.
        dict(name="packed_gdn_64", kind="packed", backbone="gdn", seqs=64, lo=100, hi=4000, mix=11, H=16),
        # One training step of the mixer at 4K (forward, then the gradients of every input).
        dict(name="train_gla_4k", kind="train", backbone="gla", B=4, T=4096, H=16),
        dict(name="train_gdn_4k", kind="train", backbone="gdn", B=4, T=4096, H=16),
        # Full-precision evaluation of a small model: fp32 inputs, two heads of 64.
        dict(name="fp32_gla_small", kind="fp32", backbone="gla", B=1, T=256, H=2, d=64),
    ]


#: Tokens times heads of the largest listed case of each kind: a drawn one has no more.
MOST = {"prefill": 8 * 4096 * 16, "packed": 64 * 2050 * 16, "train": 4 * 4096 * 16, "fp32": 4096}


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["decode", "prefill", "prefill", "prefill", "packed", "train", "train", "fp32"])
    backbone = rng.choice(["gla", "gdn"])
    if kind == "decode":
        return dict(kind=kind, backbone=backbone, B=_log_int(rng, 1, 256), H=rng.choice([4, 8, 16]),
                    d=rng.choice([64, 128, 128]))
    H = rng.choice([4, 8, 12, 16, 16])
    if kind == "prefill":
        T = _log_int(rng, 40, 20480)
        B = _log_int(rng, 1, max(1, min(32, MOST[kind] // (T * H))))
        return dict(kind=kind, backbone=backbone, B=B, T=T, H=H, resumed=rng.random() < 0.5)
    if kind == "packed":
        seqs = _log_int(rng, 3, 64)
        hi = _log_int(rng, 300, 4000)
        return dict(kind=kind, backbone=backbone, seqs=seqs, lo=_log_int(rng, 1, 100), hi=hi,
                    mix=rng.randrange(1 << 20), H=H)
    if kind == "train":
        T = _log_int(rng, 100, 8192)
        B = _log_int(rng, 1, max(1, min(16, MOST[kind] // (T * H))))
        return dict(kind=kind, backbone=backbone, B=B, T=T, H=H)
    H = rng.choice([2, 4])
    T = _log_int(rng, 30, 1000)
    return dict(kind=kind, backbone=backbone, B=_log_int(rng, 1, max(1, MOST[kind] // (T * H))), T=T, H=H,
                d=rng.choice([64, 128]))


def _lengths(case):
    r = random.Random(case["mix"])
    return [r.randint(case["lo"], case["hi"]) for _ in range(case["seqs"])]


def _unit(x):
    return x / x.norm(dim=-1, keepdim=True).clamp_min(1e-30)


def _tokens(gen, backbone, B, T, H, d, dtype):
    """q, k, v, gate, beta, lambda of the repository's input recipe, drawn on the GPU: N(0, 1) values, unit
    keys (Gated DeltaNet: queries too), log-forget gates logsigmoid(N)/16 or -softplus(N), beta = sigmoid(N), and
    the lambda statistics of a trained layer (sigmoid(N(logit 0.29, 0.5)))."""
    def n(*shape):
        return torch.randn(*shape, device="cuda", generator=gen)

    q, k, v = n(B, T, H, d), _unit(n(B, T, H, d)), n(B, T, H, d)
    if backbone == GLA:
        gate, beta = (F.logsigmoid(n(B, T, H, d)) / 16).to(dtype), None
    else:
        q = _unit(q)
        gate, beta = -F.softplus(n(B, T, H)), torch.sigmoid(n(B, T, H))
    lam = torch.sigmoid(math.log(0.29 / 0.71) + 0.5 * n(B, T, H))
    return q.to(dtype), k.to(dtype), v.to(dtype), gate, beta, lam


def _cache(gen, B, H, d, past=64):
    """The state that ``past`` tokens left: the sums of their unit keys and a fast-weight state of unit scale."""
    k = _unit(torch.randn(B, H, past, d, device="cuda", generator=gen))
    return ccq.CCQState(torch.randn(B, H, d, d, device="cuda", generator=gen) / d ** 0.5,
                        (k.transpose(-1, -2) @ k).contiguous(), k.sum(2).contiguous(),
                        torch.full((B,), past, dtype=torch.int64, device="cuda"))


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    kind, backbone, H = case["kind"], GLA if case["backbone"] == "gla" else GDN, case["H"]
    d = case.get("d", 128)
    s = {"kind": kind, "backbone": backbone, "cache": None}
    if kind == "packed":
        lens = _lengths(case)
        s["cu"] = [sum(lens[:i]) for i in range(len(lens) + 1)]
        x = _tokens(gen, backbone, 1, s["cu"][-1], H, d, torch.bfloat16)
        s["x"] = [None if t is None else t[0] for t in x]
    elif kind == "decode":
        x = _tokens(gen, backbone, case["B"], 1, H, d, torch.bfloat16)
        s["x"] = [None if t is None else t[:, 0].contiguous() for t in x]
        s["cache"] = _cache(gen, case["B"], H, d)
    else:
        s["x"] = _tokens(gen, backbone, case["B"], case["T"], H, d,
                         torch.float32 if kind == "fp32" else torch.bfloat16)
        if kind == "train":
            s["dout"] = torch.randn(case["B"], case["T"], H, d, device="cuda", generator=gen).bfloat16()
        if case.get("resumed"):
            s["cache"] = _cache(gen, case["B"], H, d)
    return s


def _state_dict(st):
    return {"S": st.S, "C": st.C, "m": st.m, "t": st.t}


def run(s):
    q, k, v, gate, beta, lam = s["x"]
    if s["kind"] == "decode":
        o = ccq.decode_step(s["backbone"], q, k, v, gate, lam, s["cache"], beta)
        return {"o": o, **_state_dict(s["cache"])}
    if s["kind"] == "packed":
        o, st = ccq.fwd_varlen(s["backbone"], q, k, v, gate, lam, s["cu"], beta=beta)
        return {"o": o, **_state_dict(st)}
    if s["kind"] == "train":
        if s["backbone"] == GLA:
            o, _, ckpt = ccq.gla_fwd_save(q, k, v, gate, lam, return_state=False)
            return {"o": o, **ccq.gla_bwd(q, k, v, gate, lam, s["dout"], ckpt=ckpt)}
        o = ccq.gdn_fwd(q, k, v, gate, beta, lam, return_state=False)
        return {"o": o, **ccq.gdn_bwd(q, k, v, gate, beta, lam, s["dout"])}
    if s["backbone"] == GLA:
        o, st = ccq.gla_fwd(q, k, v, gate, lam, s["cache"])
    else:
        o, st = ccq.gdn_fwd(q, k, v, gate, beta, lam, s["cache"])
    return {"o": o, **_state_dict(st)}


def work(case):
    """Bytes: every input, output and (initial, final) state once.  Flops: the chunk form's dense products for
    bf16 prefill and training (per 64-token chunk and head of 128: GLA 12.6 M, Gated DeltaNet 16.8 M forward,
    33.6 M more backward), the recurrence's rank-one updates and matrix-vector products otherwise."""
    kind, gla, H, d = case["kind"], case["backbone"] == "gla", case["H"], case.get("d", 128)
    size = 4 if kind == "fp32" else 2
    state = (2 * d * d + d) * 4
    gates = d * size + 4 if gla else 12
    if kind == "decode":
        n = case["B"] * H
        return {"bytes": n * (4 * d * size + gates + 2 * state), "flops": n * (8 if gla else 10) * d * d}
    if kind == "packed":
        rows, lens = case["seqs"], _lengths(case)
    else:
        rows, lens = case["B"], [case["T"]] * case["B"]
    tokens = sum(lens) * H
    out = tokens * (4 * d * size + gates)
    states = rows * H * state * (2 if case.get("resumed") else 1)
    if kind == "fp32":
        return {"bytes": out + states, "flops": tokens * (8 if gla else 10) * d * d}
    chunks = sum(-(-n // CHUNK) for n in lens) * H
    flops = chunks * (48 if gla else 64) * CHUNK ** 2 * CHUNK
    if kind == "train":
        out += tokens * (7 * d * size + 2 * gates)
        flops += chunks * 128 * CHUNK ** 3
    return {"bytes": out + states, "flops": flops}


def _forward64(backbone, q, k, v, gate, beta, lam, S, C, m, t):
    """CCQ in 64 bits, 64 tokens at a time.  Tokens [B, H, T, ...], states [B, H, ...], t [B]."""
    d = q.shape[-1]
    q = q * q.square().sum(-1, keepdim=True).clamp_min(1e-12).rsqrt()
    k = k * k.square().sum(-1, keepdim=True).clamp_min(1e-12).rsqrt()
    outs = []
    for a in range(0, q.shape[2], CHUNK):
        Q, K, V, l = (x[:, :, a:a + CHUNK] for x in (q, k, v, lam))
        n = Q.shape[2]
        pos = (t.view(-1, 1, 1) + torch.arange(a + 1, a + n + 1, device=q.device)).unsqueeze(-1).double()
        sc = (Q @ K.transpose(-1, -2)).tril()
        mean = (m.unsqueeze(2) + K.cumsum(2)) / pos
        corr = ((Q * m.unsqueeze(2)).sum(-1) + sc.sum(-1)).unsqueeze(-1) / pos
        qc = Q - l.unsqueeze(-1) * ((Q @ C.transpose(-1, -2) + sc @ K) / pos - corr * mean)
        if backbone == GLA:
            G = gate[:, :, a:a + n].cumsum(2)
            last, mid = G[:, :, -1:], G[:, :, n // 2:n // 2 + 1]
            s = ((qc * (G - mid).exp()) @ (K * (mid - G).exp()).transpose(-1, -2)).tril()
            outs.append(((qc * G.exp()) @ S + s @ V) / d ** 0.5)
            S = last.exp().transpose(-1, -2) * S + (K * (last - G).exp()).transpose(-1, -2) @ V
        else:
            g, b = gate[:, :, a:a + n].cumsum(2).unsqueeze(-1), beta[:, :, a:a + n].unsqueeze(-1)
            low = torch.ones(n, n, device=q.device, dtype=torch.bool).tril()
            dec = (g - g.transpose(-1, -2)).masked_fill(~low, -math.inf).exp()
            A = (b * dec * (K @ K.transpose(-1, -2))).tril(-1) + torch.eye(n, device=q.device, dtype=q.dtype)
            U = torch.linalg.solve_triangular(A, b * (V - g.exp() * (K @ S)), upper=False, unitriangular=True)
            outs.append(((g.exp() * qc) @ S + ((qc @ K.transpose(-1, -2)) * dec) @ U) / d ** 0.5)
            S = g[:, :, -1:].exp() * S + (K * (g[:, :, -1:] - g).exp()).transpose(-1, -2) @ U
        C = C + K.transpose(-1, -2) @ K
        m = m + K.sum(2)
    return torch.cat(outs, 2), S, C, m


def _heads_first(x):
    return None if x is None else x.double().transpose(1, 2)


def exact(case, seed):
    s = prepare(case, seed)
    backbone, c = s["backbone"], s["cache"]
    x = s["x"]
    if s["kind"] == "packed":
        parts = []
        for a, b in zip(s["cu"], s["cu"][1:]):
            parts.append(_exact_prefill(backbone, [None if y is None else y[a:b].unsqueeze(0) for y in x], None))
        out = {"o": torch.cat([p["o"][0] for p in parts])}
        return {**out, **{n: torch.cat([p[n] for p in parts]) for n in "SCmt"}}
    if s["kind"] == "decode":
        r = _exact_prefill(backbone, [None if y is None else y.unsqueeze(1) for y in x], c)
        return {**r, "o": r["o"][:, 0].contiguous()}
    if s["kind"] != "train":
        return _exact_prefill(backbone, x, c)
    B, T, H, d = x[0].shape
    leaves = [None if y is None else y.double().requires_grad_() for y in x]
    zero = [torch.zeros(B, H, *n, device="cuda", dtype=torch.double, requires_grad=True) for n in ((d, d), (d, d), (d,))]
    o = _forward64(backbone, *(None if y is None else y.transpose(1, 2) for y in leaves), *zero,
                   torch.zeros(B, device="cuda", dtype=torch.int64))[0].transpose(1, 2)
    names = ["dq", "dk", "dv", "dgk" if backbone == GLA else "dg", "dbeta", "dlambda", "dS0", "dC0", "dm0"]
    want = [(n, y) for n, y in zip(names, leaves + zero) if y is not None]
    got = torch.autograd.grad(o, [y for _, y in want], s["dout"].double())
    return {"o": o.detach().contiguous(), **{n: g.contiguous() for (n, _), g in zip(want, got)}}


def _exact_prefill(backbone, x, c):
    B, T, H, d = x[0].shape
    if c is None:
        z = dict(device="cuda", dtype=torch.double)
        S, C, m = torch.zeros(B, H, d, d, **z), torch.zeros(B, H, d, d, **z), torch.zeros(B, H, d, **z)
        t = torch.zeros(B, device="cuda", dtype=torch.int64)
    else:
        S, C, m, t = c.S.double(), c.C.double(), c.m.double(), c.t
    o, S, C, m = _forward64(backbone, *(_heads_first(y) for y in x), S, C, m, t)
    return {"o": o.transpose(1, 2).contiguous(), "S": S, "C": C, "m": m, "t": t + T}
