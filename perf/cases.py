"""Timed cases of the framework's main path, called as a user's program calls it.

A case is one layer's worth of work through the public entry points of
``paper_2607_08186_gb300.binding``: a training layer (forward and backward), a
prefill (forward only), a final-stream-only layer, a decoding step over the
expanded KV cache, or the embedding ends of a training step.  Head layouts and
lengths are the ones the repository's own configurations, tests and benchmark use.
"""
from __future__ import annotations

import math

import torch

from paper_2607_08186_gb300 import binding as hd
from paper_2607_08186_gb300.inputs import CROSS, LOCAL, WITHIN

MODES = {"within": WITHIN, "cross": CROSS, "local": LOCAL}
DEV = "cuda"

# (query heads, K/V heads, head dim): 8B-class dense, large-MoE-class, 617B grouping, 80B, and small heads
HEADS = [(32, 8, 128), (64, 8, 128), (96, 8, 128), (24, 2, 256), (16, 4, 64), (4, 4, 64)]
MAX_ATTN_FLOPS = 8.0e12    # a drawn attention case, below the largest listed one
MAX_CACHE_BYTES = 7.0e9    # a drawn cache, below the largest listed one
MAX_EXACT_FLOPS = 1.2e13   # beyond this the 64-bit reference takes too long


def _attn(name, kind, mode, B, L, n, heads, window=0):
    return {"name": name, "kind": kind, "mode": mode, "B": B, "L": L, "n": n, "Hq": heads[0], "Hkv": heads[1],
            "Dh": heads[2], "window": window}


def listed():
    return [
        # smallest: one layer of the tiny configuration (unit tests, debugging runs): launches and latency
        _attn("train_tiny_within", "train", "within", 1, 64, 2, (4, 4, 64)),
        # the benchmark layer: an intra-stream layer of the 8B-class model in training
        _attn("train_8b_within", "train", "within", 1, 4096, 4, (32, 8, 128)),
        # a cross-stream layer on a packed batch of two sequences of odd length
        _attn("train_8b_cross_ragged", "train", "cross", 2, 1021, 4, (32, 8, 128)),
        # a sliding-window layer of the 8B-class model
        _attn("train_8b_local", "train", "local", 1, 4096, 4, (32, 8, 128), 1024),
        # an intra-stream layer of the 80B configuration (head dim 256)
        _attn("train_80b_within", "train", "within", 1, 4096, 4, (24, 2, 256)),
        # one of the 80B configuration's mirrored layers: final-stream queries over all streams' keys
        _attn("final_80b_cross", "final", "cross", 1, 4096, 4, (24, 2, 256)),
        # long-context prefill of a cross-stream layer: 32768 positions, forward only (the largest)
        _attn("prefill_8b_cross_32k", "prefill", "cross", 1, 8192, 4, (32, 8, 128)),
        # batched prefill of a small model: head dim 64, odd stream count, lengths off every tile size
        _attn("prefill_dh64_ragged", "prefill", "within", 4, 1501, 3, (16, 4, 64)),
        # single-user decoding at 8k tokens: cache append and one intra-stream step
        _attn("decode_8b_b1_8k", "decode", "within", 1, 8192, 4, (32, 8, 128)),
        # a serving batch of 16 sequences of different lengths up to 32k tokens, cross-stream step
        _attn("decode_8b_b16_32k", "decode", "cross", 16, 32768, 4, (32, 8, 128)),
        # a small serving batch of the 80B configuration
        _attn("decode_80b_b4_8k", "decode", "within", 4, 8192, 4, (24, 2, 256)),
        # the embedding ends of a training step: expansion, final-stream selection and both adjoints, ids
        # repeating as in natural language
        {"name": "embed_8b", "kind": "embed", "B": 1, "L": 4096, "n": 4, "V": 151936, "D": 4096, "zipf": 1.0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["train", "train", "prefill", "final", "decode", "decode", "embed"])
    n = rng.choice([1, 2, 3, 4, 4, 8])
    if kind == "embed":
        c = {"kind": "embed", "B": rng.choice([1, 2, 3]), "L": _log_int(rng, 64, 4096), "n": min(n, 4),
             "V": _log_int(rng, 1000, 151936), "D": 8 * _log_int(rng, 32, 512), "zipf": rng.choice([0.0, 1.0])}
        while c["B"] * c["L"] > 6000:
            c["L"] //= 2
        return c
    heads = rng.choice(HEADS)
    mode = rng.choice(["within", "cross", "local"])
    B = rng.choice([1, 1, 2, 3, 4])
    if kind == "decode":
        B = rng.choice([1, 2, 4, 7, 16])
        c = _attn("", kind, mode, B, _log_int(rng, 100, 32768), n, heads)
        while 4.0 * B * c["L"] * n * heads[1] * heads[2] > MAX_CACHE_BYTES:
            c["L"] = c["L"] * 3 // 4
    else:
        c = _attn("", kind, mode, B, _log_int(rng, 64, 8192), n, heads)
        while work(c)["flops"] > MAX_ATTN_FLOPS or B * c["L"] * n * heads[0] * heads[2] > 2.7e8:
            c["L"] = c["L"] * 3 // 4
    if mode == "local":
        c["window"] = _log_int(rng, 16, 4096)
    del c["name"]
    return c


# ------------------------------------------------------------------ state

class State:
    pass


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed * 7919 + 17)


def _randn(g, *shape, std=1.0, dtype=torch.bfloat16):
    x = torch.empty(shape, dtype=dtype, device=DEV)
    x.normal_(0.0, std, generator=g)
    return x


def _lens(c):
    """Tokens in each sequence's cache: the first fills it, the others spread over a quarter to all of it."""
    return [c["L"]] + [max(1, int(c["L"] * (0.25 + 0.75 * (0.6180339887 * b % 1.0)))) for b in range(1, c["B"])]


def _token_ids(c, g):
    if c["zipf"] <= 0:
        return torch.randint(0, c["V"], (c["B"], c["L"]), generator=g, device=DEV, dtype=torch.int32)
    w = torch.arange(1, c["V"] + 1, dtype=torch.float64, device=DEV).pow(-c["zipf"])
    return torch.multinomial(w, c["B"] * c["L"], replacement=True, generator=g).view(c["B"], c["L"]).to(torch.int32)


def prepare(case, seed):
    s, g = State(), _gen(seed)
    s.case = c = dict(case)
    s.status = torch.zeros(1, dtype=torch.int32, device=DEV)
    B, L, n = c["B"], c["L"], c["n"]
    if c["kind"] == "embed":
        V, D = c["V"], c["D"]
        s.tables = _randn(g, n, V, D, std=0.02)
        s.ids = _token_ids(c, g)
        s.x = torch.empty(B, n * L, D, dtype=torch.bfloat16, device=DEV)
        s.y = torch.empty(B, L, D, dtype=torch.bfloat16, device=DEV)
        s.dy = _randn(g, B, L, D)
        s.dh = torch.empty(B, n * L, D, dtype=torch.bfloat16, device=DEV)
        s.dx = _randn(g, B, n * L, D)  # the gradient that reaches the embeddings through the layers
        # gradient accumulation: the tables' gradients already hold an earlier micro-batch
        s.dtables = _randn(g, n, V, D, dtype=torch.float32)
        s.ws = torch.empty(hd.hd_expand_embed_bwd_workspace_bytes(B, L), dtype=torch.uint8, device=DEV)
        return s
    Hq, Hkv, Dh = c["Hq"], c["Hkv"], c["Dh"]
    s.mode = MODES[c["mode"]]
    if c["kind"] == "decode":
        s.q = _randn(g, B, n, Hq, Dh)
        s.kn, s.vn = _randn(g, B, n, Hkv, Dh), _randn(g, B, n, Hkv, Dh)
        s.kc, s.vc = _randn(g, B, L * n, Hkv, Dh), _randn(g, B, L * n, Hkv, Dh)
        s.lens = torch.tensor(_lens(c), dtype=torch.int32, device=DEV)
        s.o = torch.empty_like(s.q)
        s.lse = torch.empty(B, Hq, n, dtype=torch.float32, device=DEV)
        s.ws = torch.empty(hd.sfa_decode_workspace_bytes(B, L, n, Hq, Hkv, Dh, s.mode, c["window"]),
                           dtype=torch.uint8, device=DEV)
        return s
    Lq = L if c["kind"] == "final" else n * L
    s.q = _randn(g, B, Lq, Hq, Dh)
    s.k, s.v = _randn(g, B, n * L, Hkv, Dh), _randn(g, B, n * L, Hkv, Dh)
    s.o = torch.empty_like(s.q)
    s.lse = torch.empty(B, Hq, Lq, dtype=torch.float32, device=DEV)
    if c["kind"] != "prefill":
        s.do = _randn(g, B, Lq, Hq, Dh)
        s.dq, s.dk, s.dv = torch.empty_like(s.q), torch.empty_like(s.k), torch.empty_like(s.v)
        ws_bytes = hd.sfa_bwd_final_workspace_bytes if c["kind"] == "final" else hd.sfa_bwd_workspace_bytes
        s.ws = torch.empty(ws_bytes(B, L, n, Hq, Hkv, Dh, s.mode), dtype=torch.uint8, device=DEV)
    return s


def run(s):
    c = s.case
    kind, n = c["kind"], c["n"]
    if kind == "train":
        hd.sfa_fwd(s.q, s.k, s.v, s.o, s.lse, n, s.mode, window=c["window"], dev_status=s.status)
        hd.sfa_bwd(s.q, s.k, s.v, s.o, s.lse, s.do, s.dq, s.dk, s.dv, n, s.mode, s.ws, window=c["window"],
                   dev_status=s.status)
        return {"o": s.o, "lse": s.lse, "dq": s.dq, "dk": s.dk, "dv": s.dv, "status": s.status}
    if kind == "prefill":
        hd.sfa_fwd(s.q, s.k, s.v, s.o, s.lse, n, s.mode, window=c["window"], dev_status=s.status)
        return {"o": s.o, "lse": s.lse, "status": s.status}
    if kind == "final":
        hd.sfa_fwd_final(s.q, s.k, s.v, s.o, s.lse, s.mode, window=c["window"], dev_status=s.status)
        hd.sfa_bwd_final(s.q, s.k, s.v, s.o, s.lse, s.do, s.dq, s.dk, s.dv, s.mode, s.ws, window=c["window"],
                         dev_status=s.status)
        return {"o": s.o, "lse": s.lse, "dq": s.dq, "dk": s.dk, "dv": s.dv, "status": s.status}
    if kind == "decode":
        hd.sfa_kv_append(s.kn, s.vn, s.kc, s.vc, s.lens, n, dev_status=s.status)
        hd.sfa_decode(s.q, s.kc, s.vc, s.lens, s.o, n, s.mode, s.ws, lse=s.lse, window=c["window"],
                      dev_status=s.status)
        return {"o": s.o, "lse": s.lse, "k_cache": s.kc, "v_cache": s.vc, "status": s.status}
    hd.hd_expand_embed(s.tables, s.ids, s.x, dev_status=s.status)
    hd.hd_select_final_stream(s.x, s.y, n)
    hd.hd_select_final_stream_bwd(s.dy, s.dh, n)
    hd.hd_expand_embed_bwd(s.dx, s.ids, s.dtables, s.ws, dev_status=s.status)
    return {"x": s.x, "y": s.y, "dh": s.dh, "dtables": s.dtables, "status": s.status}


# ------------------------------------------------------------------ work

def _visible_pairs(c):
    """Visible (query, key) pairs of one query head over the whole batch."""
    B, L, n, w = c["B"], c["L"], c["n"], c["window"]
    N = n * L

    def local(p):
        return min(p + 1, w)

    if c["kind"] == "decode":
        if c["mode"] == "within":
            return n * sum(_lens(c))
        if c["mode"] == "cross":
            return sum((T - 1) * n + s + 1 for T in _lens(c) for s in range(n))
        return sum(local((T - 1) * n + s) for T in _lens(c) for s in range(n))
    if c["kind"] == "final":
        if c["mode"] == "within":
            return B * L * (L + 1) // 2
        if c["mode"] == "cross":
            return B * n * L * (L + 1) // 2
        return B * sum(local(t * n + n - 1) for t in range(L))
    if c["mode"] == "within":
        return B * n * L * (L + 1) // 2
    if c["mode"] == "cross":
        return B * N * (N + 1) // 2
    m = min(w, N)
    return B * (m * (m + 1) // 2 + (N - m) * m)


def work(case):
    c = case
    B, L, n = c["B"], c["L"], c["n"]
    if c["kind"] == "embed":
        V, D, N = c["V"], c["D"], c["B"] * c["L"]
        if c["zipf"] > 0:
            w = torch.arange(1, V + 1, dtype=torch.float64).pow(-c["zipf"])
            p = w / w.sum()
        else:
            p = torch.full((V,), 1.0 / V, dtype=torch.float64)
        distinct = float((1.0 - (1.0 - p).pow(N)).sum())
        rows = 2 * D
        gather = n * (distinct + N) * rows + 4 * N
        select = 2 * N * rows + N * rows + n * N * rows
        bwd = n * N * rows + n * distinct * D * 8 + 4 * N
        return {"bytes": gather + select + bwd, "flops": float(n * N * D)}
    Hq, Hkv, Dh = c["Hq"], c["Hkv"], c["Dh"]
    pairs = _visible_pairs(c)
    if c["kind"] == "decode":
        keys = sum(min(n * T, c["window"] + n - 1) if c["mode"] == "local" else n * T for T in _lens(c))
        bytes_ = keys * Hkv * Dh * 4 + B * (2 * n * Hq * Dh * 2 + n * Hkv * Dh * 8 + n * Hq * 4)
        return {"bytes": float(bytes_), "flops": 4.0 * Dh * Hq * pairs}
    Lq = L if c["kind"] == "final" else n * L
    qb, kb = B * Lq * Hq * Dh * 2, B * n * L * Hkv * Dh * 2
    fwd = 2 * qb + 2 * kb + B * Lq * Hq * 4
    if c["kind"] == "prefill":
        return {"bytes": float(fwd), "flops": 4.0 * Dh * Hq * pairs}
    return {"bytes": float(fwd + 4 * qb + 4 * kb + B * Lq * Hq * 4), "flops": 14.0 * Dh * Hq * pairs}


# ------------------------------------------------------------------ 64-bit reference

def _positions(c, s):
    """Position of each query row and each key row, on the device."""
    N, n = c["n"] * c["L"], c["n"]
    kp = torch.arange(N, device=DEV)
    if c["kind"] == "final":
        return torch.arange(c["L"], device=DEV) * n + n - 1, kp
    if c["kind"] == "decode":
        return None, kp
    return kp, kp


def _visible(c, qp, kp):
    vis = kp[None, :] <= qp[:, None]
    if c["mode"] == "local":
        vis &= kp[None, :] > qp[:, None] - c["window"]
    if c["mode"] == "within":
        vis &= (kp[None, :] % c["n"]) == (qp[:, None] % c["n"])
    return vis


def _problems(c, qp, kp):
    """(query rows, key rows) index tensors that cover every visible pair: one per stream where streams do not mix."""
    n = c["n"]
    if c["mode"] != "within":
        return [(torch.arange(len(qp), device=DEV), torch.arange(len(kp), device=DEV))]
    out = []
    for s in range(n):
        qi, ki = (qp % n == s).nonzero().flatten(), (kp % n == s).nonzero().flatten()
        if len(qi):
            out.append((qi, ki))
    return out


def _exact_group(c, q, k, v, do, qp, kp, o, lse, dq, dk, dv):
    """One sequence and K/V head: q, do [G][Lq][Dh], k, v [Lk][Dh], all float64; results are written in place."""
    scale = 1.0 / math.sqrt(c["Dh"])
    for qi, ki in _problems(c, qp, kp):
        kpi = kp[ki]
        step = 1024
        for a in range(0, len(qi), step):
            rows = qi[a:a + step]
            pos = qp[rows]
            lo = 0
            if c["mode"] == "local":
                lo = int(torch.searchsorted(kpi, torch.clamp(pos[0] - c["window"] + 1, min=0)))
            hi = int(torch.searchsorted(kpi, pos[-1], right=True))
            cols = ki[lo:hi]
            kk, vv = k[cols], v[cols]
            z = torch.matmul(q[:, rows], kk.T).mul_(scale)
            z.masked_fill_(~_visible(c, pos, kpi[lo:hi])[None], -math.inf)
            ls = torch.logsumexp(z, dim=-1)
            p = z.sub_(ls[..., None]).exp_()
            ob = torch.matmul(p, vv)
            o[:, rows], lse[:, rows] = ob, ls
            if do is None:
                continue
            d = do[:, rows]
            dv[cols] += torch.einsum("gqk,gqd->kd", p, d)
            ds = torch.matmul(d, vv.T).sub_((d * ob).sum(-1)[..., None]).mul_(p)
            dq[:, rows] = torch.matmul(ds, kk).mul_(scale)
            dk[cols] += torch.einsum("gqk,gqd->kd", ds, q[:, rows]).mul_(scale)


def exact(case, seed):
    c = case
    if c["kind"] != "embed" and work(c)["flops"] > MAX_EXACT_FLOPS:
        return None
    s = prepare(c, seed)
    B, L, n = c["B"], c["L"], c["n"]
    if c["kind"] == "embed":
        ids = s.ids.long().flatten()
        x = torch.stack([s.tables[i][ids] for i in range(n)], 1).view(B, n * L, -1)
        dh = torch.zeros_like(s.dh)
        dh[:, n - 1::n] = s.dy
        dt = s.dtables.double()
        for i in range(n):
            dt[i].index_add_(0, ids, s.dx[:, i::n].reshape(B * L, -1).double())
        return {"x": x, "y": x[:, n - 1::n].contiguous(), "dh": dh, "dtables": dt, "status": s.status}
    Hq, Hkv, Dh = c["Hq"], c["Hkv"], c["Dh"]
    G = Hq // Hkv
    if c["kind"] == "decode":
        o = torch.zeros(B, n, Hq, Dh, dtype=torch.float64, device=DEV)
        lse = torch.zeros(B, Hq, n, dtype=torch.float64, device=DEV)
        for b in range(B):
            T = int(s.lens[b])
            s.kc[b, (T - 1) * n:T * n], s.vc[b, (T - 1) * n:T * n] = s.kn[b], s.vn[b]
            qp, kp = torch.arange((T - 1) * n, T * n, device=DEV), torch.arange(T * n, device=DEV)
            vis = _visible(c, qp, kp)
            for h in range(Hkv):
                k, v = s.kc[b, :T * n, h].double(), s.vc[b, :T * n, h].double()
                q = s.q[b, :, h * G:(h + 1) * G].double()  # [n][G][Dh]
                z = torch.matmul(q, k.T).div_(math.sqrt(Dh)).masked_fill_(~vis[:, None], -math.inf)
                ls = torch.logsumexp(z, dim=-1)
                o[b, :, h * G:(h + 1) * G] = torch.matmul(torch.exp(z - ls[..., None]), v)
                lse[b, h * G:(h + 1) * G] = ls.T
        return {"o": o, "lse": lse, "k_cache": None, "v_cache": None, "status": s.status}
    qp, kp = _positions(c, s)
    grad = c["kind"] != "prefill"
    o = torch.zeros(s.q.shape, dtype=torch.float64, device=DEV)
    lse = torch.zeros(s.lse.shape, dtype=torch.float64, device=DEV)
    dq = torch.zeros(s.q.shape, dtype=torch.float64, device=DEV) if grad else None
    dk = torch.zeros(s.k.shape, dtype=torch.float64, device=DEV) if grad else None
    dv = torch.zeros(s.k.shape, dtype=torch.float64, device=DEV) if grad else None
    for b in range(B):
        for h in range(Hkv):
            hs = slice(h * G, (h + 1) * G)
            q = s.q[b, :, hs].transpose(0, 1).double()
            do = s.do[b, :, hs].transpose(0, 1).double() if grad else None
            ob, lb = torch.zeros_like(q), torch.zeros(q.shape[:2], dtype=torch.float64, device=DEV)
            dqb = torch.zeros_like(q) if grad else None
            _exact_group(c, q, s.k[b, :, h].double(), s.v[b, :, h].double(), do, qp, kp, ob, lb, dqb,
                         dk[b, :, h] if grad else None, dv[b, :, h] if grad else None)
            o[b, :, hs], lse[b, hs] = ob.transpose(0, 1), lb
            if grad:
                dq[b, :, hs] = dqb.transpose(0, 1)
    if not grad:
        return {"o": o, "lse": lse, "status": s.status}
    return {"o": o, "lse": lse, "dq": dq, "dk": dk, "dv": dv, "status": s.status}
