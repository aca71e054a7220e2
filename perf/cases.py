"""The work that programs have this library do, as measurable cases.

A case is a dict of plain values: its ``kind`` names the entry point, the rest
are sizes.  Shapes are those of the workloads in ``inputs.py`` (the 70M- to
1B-parameter decoder shapes, head dimension 64) and of the tests; ``draw``
spreads over the ranges between and around them.

A cache in a decode, chunk or append case is one that a serving program holds:
its pages were assigned earlier (in order, or shuffled as after many requests
came and went) and hold bottleneck vectors of unit variance, its ring holds the
window's keys and values.  Cases that append set the lengths back first, as a
program does that gives the slots to new requests or drops drafted tokens, so
every pass does the same amount of work.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import torch

from paper_2606_18587_gb300 import dar

D_HEAD = 64
PAGE = dar.PAGE_SIZE
DTYPE = {"f32": torch.float32, "bf16": torch.bfloat16}


# ----------------------------------------------------------------------- cases


def listed():
    return [
        # one short chat turn on the smallest model: a token joins a context that still fits the window
        dict(name="step_70m_b1", kind="step", dtype="bf16", B=1, Hq=8, Hkv=8, Lmin=100, Lmax=100, w=128, dd=16,
             shuffled=False),
        # batched serving of the 160M shape: append one token to each sequence and attend (the benchmark's step)
        dict(name="step_160m", kind="step", dtype="bf16", B=32, Hq=12, Hkv=12, Lmin=4096, Lmax=4096, w=128, dd=16,
             shuffled=False),
        # grouped-query serving of the 1B shape with ragged contexts and recycled pages
        dict(name="decode_1b_gqa", kind="decode", dtype="bf16", B=64, Hq=32, Hkv=8, Lmin=1024, Lmax=32768, w=256,
             dd=16, shuffled=True, direct=False),
        # a long-context point of the window x d_down sweep: wide window, wide bottleneck
        dict(name="decode_sweep_w1024_dd32", kind="decode", dtype="bf16", B=16, Hq=16, Hkv=16, Lmin=16384,
             Lmax=16384, w=1024, dd=32, shuffled=False, direct=False),
        # prompt processing / evaluation of the 410M shape at its full batch
        dict(name="prefill_410m", kind="prefill", dtype="bf16", B=8, Hq=16, Hkv=16, N=8192, w=512, dd=16,
             direct=False),
        # the smallest forward, in full precision: reference runs and gradient checks
        dict(name="prefill_f32_tiny", kind="prefill", dtype="f32", B=1, Hq=4, Hkv=4, N=256, w=32, dd=16,
             direct=False),
        # a training micro-batch of the 70M shape: sequences of 2048 tokens predict their last 2047
        dict(name="train_70m", kind="train", dtype="bf16", B=8, Hq=8, Hkv=8, N=2047, w=128, dd=16),
        # a training micro-batch of the 410M shape at long context
        dict(name="train_410m", kind="train", dtype="bf16", B=8, Hq=16, Hkv=16, N=8192, w=512, dd=16),
        # a batch of prompts of different lengths enters an empty 160M cache
        dict(name="append_prompts_160m", kind="append", dtype="bf16", B=32, Hkv=12, Nmin=1000, N=4096, w=128, dd=16,
             shuffled=False),
        # long prompts of the 1B shape enter their caches chunk by chunk
        dict(name="chunk_1b_gqa", kind="chunk", dtype="bf16", B=4, Hq=32, Hkv=8, N=512, Lmin=2048, Lmax=8000, w=256,
             dd=16, shuffled=True),
        # the latent form (one bottleneck per token for all heads): ragged grouped-query serving
        dict(name="latent_decode_1b", kind="latent_decode", dtype="bf16", B=64, Hq=32, Hkv=8, D=2048, dl=256,
             Lmin=1024, Lmax=8192, w=256, shuffled=True),
        # the latent form: prompts of different lengths enter the cache through W_down
        dict(name="latent_append_1b", kind="latent_append", dtype="bf16", B=8, Hkv=8, D=2048, dl=256, Nmin=500,
             N=1000, w=256, shuffled=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _heads(rng, most=32):
    while True:
        Hkv, G = rng.choice((1, 2, 4, 8, 12, 16)), rng.choice((1, 1, 1, 2, 4, 8))
        if Hkv * G <= most:
            return Hkv * G, Hkv


def draw(rng):
    kind = rng.choice(("step", "step", "decode", "decode", "prefill", "prefill", "train", "train", "append", "chunk",
                       "latent_decode", "latent_append"))
    dd = rng.choice((8, 16, 16, 16, 32, 64))
    w = _log(rng, 16, 1024)
    if kind in ("step", "decode"):
        Hq, Hkv = _heads(rng)
        B, Lmax = _log(rng, 1, 64), _log(rng, 40, 32768)
        Lmin = Lmax if rng.random() < 0.5 else max(1, int(Lmax * rng.uniform(0.05, 0.9)))
        while B > 1 and B * Hkv * (min(w, Lmax) * D_HEAD + Lmax * dd) * 4 > 1.0e9:  # the sweep's largest call
            B = B // 2
        c = dict(kind=kind, dtype="bf16", B=B, Hq=Hq, Hkv=Hkv, Lmin=Lmin, Lmax=Lmax, w=w, dd=dd,
                 shuffled=rng.random() < 0.5)
        if kind == "decode":
            c["direct"] = rng.random() < 0.25
        return c
    if kind in ("prefill", "train"):
        Hq, Hkv = _heads(rng, 16)
        f32 = rng.random() < 0.2
        B, N = (_log(rng, 1, 2), _log(rng, 60, 700)) if f32 else (_log(rng, 1, 8), _log(rng, 100, 8192))
        if kind == "train" and not f32:
            dd = rng.choice((16, 16, 32, 64))
        while B > 1 and B * Hq * N * N * max(dd, 16) > 8 * 16 * 8192 * 8192 * 16 / 3:
            B = B // 2
        c = dict(kind=kind, dtype="f32" if f32 else "bf16", B=B, Hq=Hq, Hkv=Hkv, N=N, w=w, dd=dd)
        if kind == "prefill":
            c["direct"] = rng.random() < 0.25
        return c
    if kind == "append":
        N = _log(rng, 2, 4096)
        return dict(kind=kind, dtype="bf16", B=_log(rng, 1, 32), Hkv=rng.choice((1, 4, 8, 12, 16)),
                    Nmin=max(1, int(N * rng.uniform(0.1, 1.0))), N=N, w=w, dd=dd, shuffled=rng.random() < 0.5)
    if kind == "chunk":
        Hq, Hkv = _heads(rng)
        Lmax = _log(rng, 64, 8192)
        return dict(kind=kind, dtype="bf16", B=_log(rng, 1, 4), Hq=Hq, Hkv=Hkv, N=_log(rng, 16, 1024),
                    Lmin=int(Lmax * rng.uniform(0.0, 1.0)), Lmax=Lmax, w=w, dd=max(dd, 16),
                    shuffled=rng.random() < 0.5)
    D, dl = rng.choice(((512, 64), (512, 128), (768, 192), (1024, 256), (2048, 256), (2048, 128)))
    if kind == "latent_decode":
        Hq, Hkv = _heads(rng)
        Lmax = _log(rng, 60, 8192)
        return dict(kind=kind, dtype="bf16", B=_log(rng, 1, 64), Hq=Hq, Hkv=Hkv, D=D, dl=dl,
                    Lmin=max(1, int(Lmax * rng.uniform(0.1, 1.0))), Lmax=Lmax, w=w, shuffled=rng.random() < 0.5)
    N = _log(rng, 1, 1000)
    return dict(kind=kind, dtype="bf16", B=_log(rng, 1, 8), Hkv=rng.choice((1, 4, 8, 12, 16)), D=D, dl=dl,
                Nmin=max(1, int(N * rng.uniform(0.3, 1.0))), N=N, w=w, shuffled=rng.random() < 0.5)


def _spread(lo, hi, n):
    """n whole numbers spread over [lo, hi] in no particular order (multiples of the golden ratio)."""
    if lo == hi:
        return [lo] * n
    return [lo + int(math.modf((i + 1) * 0.6180339887498949)[0] * (hi - lo + 1)) for i in range(n)]


def _lengths(case):
    """Tokens each sequence holds before the call."""
    if "Lmax" not in case:
        return [0] * case["B"]
    return _spread(case["Lmin"], case["Lmax"], case["B"])


def _counts(case):
    """Tokens each sequence appends in the call."""
    if case["kind"] == "step":
        return [1] * case["B"]
    if case["kind"] in ("append", "latent_append"):
        n = _spread(case["Nmin"], case["N"], case["B"])
        n[-1] = case["N"]
        return n
    return [case["N"] if case["kind"] == "chunk" else 0] * case["B"]


# ---------------------------------------------------------------------- inputs


def _normal(g, shape, std=1.0, dtype=torch.bfloat16):
    return torch.empty(shape, dtype=dtype, device="cuda").normal_(0.0, std, generator=g)


def _projections(g, Hkv, dd):
    """W_down ~ N(0, 1/d) and W_up ~ N(0, 1/d_down) of keys and values, per KV head."""
    down, up = (Hkv, D_HEAD, dd), (Hkv, dd, D_HEAD)
    f = torch.float32
    return dict(Dk=_normal(g, down, D_HEAD ** -0.5, f), Uk=_normal(g, up, dd ** -0.5, f),
                Dv=_normal(g, down, D_HEAD ** -0.5, f), Uv=_normal(g, up, dd ** -0.5, f))


def _block_table(case, paged, seed):
    """Pages for ``paged[b]`` tokens of each sequence: (table [B, most], number of pages)."""
    pages = [-(-max(0, n) // PAGE) for n in paged]
    total = max(1, sum(pages))
    ids = torch.randperm(total, generator=torch.Generator().manual_seed(seed)) if case["shuffled"] \
        else torch.arange(total)
    table = torch.full((len(pages), max(1, max(pages))), -1, dtype=torch.int32)
    at = 0
    for b, n in enumerate(pages):
        table[b, :n] = ids[at:at + n]
        at += n
    return table, total


def prepare(case, seed):
    torch.cuda.set_device(0)
    g = torch.Generator(device="cuda").manual_seed(seed)
    kind, dt = case["kind"], DTYPE[case["dtype"]]
    s = SimpleNamespace(case=case, kind=kind)
    if kind in ("prefill", "train"):
        B, Hq, Hkv, N, dd = (case[n] for n in ("B", "Hq", "Hkv", "N", "dd"))
        s.q = _normal(g, (B, Hq, N, D_HEAD), dtype=dt)
        s.k, s.v = (_normal(g, (B, Hkv, N, D_HEAD), dtype=dt) for _ in range(2))
        s.p = _projections(g, Hkv, dd)
        s.qd = _normal(g, (B, Hq, N, dd), dtype=dt) if case.get("direct") else None
        s.out = torch.empty_like(s.q)
        s.workspace = torch.empty(dar.dar_prefill_workspace_bytes(dt, B, Hkv, N, dd), dtype=torch.uint8,
                                  device="cuda")
        if kind == "train":
            s.dout = _normal(g, s.q.shape, dtype=dt)
            s.bwd_workspace = torch.empty(dar.dar_attn_backward_workspace_bytes(dt, B, Hq, Hkv, N, dd),
                                          dtype=torch.uint8, device="cuda")
            s.grads = dict(dq=torch.empty_like(s.q), dk=torch.empty_like(s.k), dv=torch.empty_like(s.v),
                           **{"d" + n: torch.empty_like(t) for n, t in s.p.items()})
        return s
    B, Hkv, w = case["B"], case["Hkv"], case["w"]
    before, new = _lengths(case), _counts(case)
    after = [a + n for a, n in zip(before, new)]
    s.lens = torch.tensor(before, dtype=torch.int32, device="cuda")
    if kind in ("latent_decode", "latent_append"):
        D, dl = case["D"], case["dl"]
        table, pages = _block_table(case, after, seed)
        s.cache = dar.DarLatentCache(B, Hkv, D, dl, w, table.shape[1], pages, block_table=table)
        s.cache.pool_c.normal_(generator=g)
    else:
        table, pages = _block_table(case, [a - w for a in after], seed)
        s.cache = dar.DarCache(B, Hkv, case["dd"], w, table.shape[1], pages, dtype=dt, block_table=table)
        s.cache.pool_kd.normal_(generator=g)
        s.cache.pool_vd.normal_(generator=g)
        s.p = _projections(g, Hkv, case["dd"])
    s.cache.win_k.normal_(generator=g)
    s.cache.win_v.normal_(generator=g)
    s.cache.seq_lens.copy_(s.lens)
    n = max(new)
    if n:
        s.k, s.v = (_normal(g, (B, Hkv, n, D_HEAD), dtype=dt) for _ in range(2))
        s.counts = torch.tensor(new, dtype=torch.int32, device="cuda") if min(new) < n else None
    if kind in ("step", "decode"):
        s.q = _normal(g, (B, case["Hq"], D_HEAD), dtype=dt)
        s.qd = _normal(g, (B, case["Hq"], case["dd"]), dtype=dt) if case.get("direct") else None
        s.workspace = dar.decode_workspace(s.cache, case["Hq"])
    elif kind == "chunk":
        s.q = _normal(g, (B, case["Hq"], n, D_HEAD), dtype=dt)
        s.workspace = torch.empty(dar.dar_prefill_chunk_workspace_bytes(s.cache, n), dtype=torch.uint8,
                                  device="cuda")
    elif kind == "latent_decode":
        s.q = _normal(g, (B, case["Hq"], D_HEAD))
        W_up = _normal(g, (dl, D), dl ** -0.5, torch.float32)
        W_K, W_V = (_normal(g, (Hkv, D, D_HEAD), D ** -0.5, torch.float32) for _ in range(2))
        s.A_K, s.A_V = dar.dar_latent_absorb(W_up, W_K, W_V)
        s.W = (W_up, W_K, W_V)
        s.workspace = dar.latent_decode_workspace(s.cache, case["Hq"])
    elif kind == "latent_append":
        s.h = _normal(g, (B, n, D))
        s.W_down = _normal(g, (D, dl), D ** -0.5, torch.float32)
    if hasattr(s, "q"):
        s.out = torch.empty_like(s.q)
    return s


def _held(c):
    """What a cache holds after a call that appends."""
    held = dict(win_k=c.win_k, win_v=c.win_v, seq_lens=c.seq_lens)
    held.update(dict(pool_c=c.pool_c) if isinstance(c, dar.DarLatentCache)
                else dict(pool_kd=c.pool_kd, pool_vd=c.pool_vd))
    return held


def run(s):
    kind, c = s.kind, s.case
    if kind == "step":
        p = s.p
        s.cache.seq_lens.copy_(s.lens)
        dar.dar_decode_step(s.cache, s.k, s.v, p["Dk"], p["Dv"], s.q, p["Uk"], p["Uv"], s.workspace, out=s.out)
        return dict(out=s.out, **_held(s.cache))
    if kind == "decode":
        if c["direct"]:
            return dar.dar_attn_decode_direct(s.cache, s.q, s.qd, s.p["Uv"], s.workspace, out=s.out)
        return dar.dar_attn_decode(s.cache, s.q, s.p["Uk"], s.p["Uv"], s.workspace, out=s.out)
    if kind == "prefill" and c["direct"]:
        return dar.dar_attn_prefill_direct(s.q, s.qd, s.k, s.v, s.p["Dk"], s.p["Dv"], s.p["Uv"], c["w"], out=s.out,
                                           workspace=s.workspace)
    if kind in ("prefill", "train"):
        args = (s.q, s.k, s.v, s.p["Dk"], s.p["Uk"], s.p["Dv"], s.p["Uv"])
        dar.dar_attn_prefill(*args, c["w"], out=s.out, workspace=s.workspace)
        if kind == "prefill":
            return s.out
        g = dar.dar_attn_backward(*args, s.out, s.dout, c["w"], workspace=s.bwd_workspace, grads=s.grads)
        return dict(out=s.out, **g)
    if kind == "latent_decode":
        return dar.dar_latent_decode(s.cache, s.q, s.A_K, s.A_V, s.workspace, out=s.out)
    s.cache.seq_lens.copy_(s.lens)
    if kind == "append":
        dar.dar_cache_append(s.cache, s.k, s.v, s.p["Dk"], s.p["Dv"], n_per_seq=s.counts)
        return _held(s.cache)
    if kind == "chunk":
        dar.dar_prefill_chunk(s.cache, s.q, s.k, s.v, s.p["Dk"], s.p["Uk"], s.p["Dv"], s.p["Uv"], out=s.out,
                              workspace=s.workspace)
        return dict(out=s.out, **_held(s.cache))
    if kind == "latent_append":
        dar.dar_latent_append(s.cache, s.h, s.k, s.v, s.W_down, n_per_seq=s.counts)
        return _held(s.cache)
    raise ValueError(kind)


# ------------------------------------------------------------- necessary work


def _pairs(L0, n, w):
    """(local, global) query-key pairs of queries at positions L0 .. L0 + n - 1."""
    full = (L0 + n) * (L0 + n + 1) // 2 - L0 * (L0 + 1) // 2
    short = max(0, min(L0 + n, w) - L0)  # queries that see fewer than w tokens
    local = (n - short) * w + short * L0 + short * (short + 1) // 2
    return local, full - local


def work(case):
    kind, Hkv, w = case["kind"], case["Hkv"], case["w"]
    e = 4 if case["dtype"] == "f32" else 2
    row = D_HEAD * e
    before, new = _lengths(case) if kind not in ("prefill", "train") else [0] * case["B"], None
    nbytes = flops = 0
    if kind in ("prefill", "train"):
        B, Hq, N, dd = (case[n] for n in ("B", "Hq", "N", "dd"))
        loc, glob = _pairs(0, N, w)
        lift = 2 * D_HEAD * dd
        nbytes = B * N * row * (2 * Hq + 2 * Hkv) + 4 * Hkv * D_HEAD * dd * 4
        flops = B * Hq * (loc * 4 * D_HEAD + glob * 4 * dd + 2 * N * lift) + 2 * B * Hkv * N * lift
        if case.get("direct"):
            nbytes += B * Hq * N * dd * e
        if kind == "train":  # dout in; dq, dk, dv and the four projections' gradients out
            nbytes += B * N * row * (2 * Hq + 2 * Hkv) + 4 * Hkv * D_HEAD * dd * 4
            flops += B * Hq * (loc * 10 * D_HEAD + glob * 12 * dd + 5 * N * lift) + 4 * B * Hkv * N * lift
        return dict(bytes=nbytes, flops=flops)
    new = _counts(case)
    if kind in ("latent_append", "latent_decode"):
        dl, D = case["dl"], case["D"]
        for L, n in zip(before, new):
            if kind == "latent_append":
                nbytes += n * D * e + n * dl * e + 4 * Hkv * min(n, w) * row
                flops += 2 * n * D * dl
            else:
                near = min(L, w)
                nbytes += 2 * Hkv * near * row + (L - near) * dl * e + 2 * case["Hq"] * row
                flops += case["Hq"] * (4 * near * D_HEAD + 4 * (L - near) * dl + 4 * D_HEAD * dl)
        nbytes += D * dl * 4 if kind == "latent_append" else 2 * Hkv * D_HEAD * dl * 4
        return dict(bytes=nbytes, flops=flops)
    dd = case["dd"]
    small = dd * e
    for L, n in zip(before, new):
        out_of_window = max(0, L + n - w) - max(0, L - w)
        from_ring = min(out_of_window, min(L, w))
        if n:  # new tokens in, ring rows that leave in, bottleneck rows and the new ring rows out
            nbytes += 2 * Hkv * (n * row + from_ring * row + out_of_window * small + min(n, w) * row)
            flops += 2 * Hkv * out_of_window * 2 * D_HEAD * dd
        if kind in ("step", "decode"):
            near = min(L + n, w)
            far = L + n - near
            nbytes += 2 * Hkv * (near * row + far * small) + 2 * case["Hq"] * row
            flops += case["Hq"] * (4 * near * D_HEAD + 4 * far * dd + 4 * D_HEAD * dd)
        elif kind == "chunk":
            loc, glob = _pairs(L, n, w)
            nbytes += 2 * Hkv * (min(L, w) * row + max(0, L - w) * small) + 2 * case["Hq"] * n * row
            flops += case["Hq"] * (4 * loc * D_HEAD + 4 * glob * dd + 4 * n * D_HEAD * dd)
    nbytes += (2 if kind == "append" else 4) * Hkv * D_HEAD * dd * 4
    return dict(bytes=nbytes, flops=flops)


def tolerance(case):
    """About four times the distance from the 64-bit result that each path shows (2-norm): decode 2e-3 to 3e-3,
    forward 3.7e-3, chunks and gradients 5e-3 to 5.5e-3 in bf16, where the output's own rounding is 1.7e-3; below
    1e-6 in fp32.  What an append writes is defined bit for bit (one fp32 chain per element, rounded once)."""
    if case["kind"] in ("append", "latent_append"):
        return "exact"
    if case["dtype"] == "f32":
        return {"rel": 4e-6}
    return {"rel": {"step": 1e-2, "decode": 1e-2, "latent_decode": 1e-2, "prefill": 1.5e-2}.get(case["kind"], 2e-2)}


# ------------------------------------------------------------ the same in 64 bits


def _attend(q, k, v, qt, kd, vd, Uv, row0, w, scale, key0):
    """Rows row0.. of the two-segment attention: q [..,n,64] and qt [..,n,dd] against full-width keys at
    positions key0.. (those within the window of each row) and bottleneck keys at positions 0.. (the others).
    Returns the output, the weights of both segments and the bottleneck value sum."""
    rows = row0 + torch.arange(q.shape[-2], device=q.device)[:, None]
    near = key0 + torch.arange(k.shape[-2], device=q.device)[None, :]
    far = torch.arange(kd.shape[-2], device=q.device)[None, :]
    S = torch.cat(((q @ k.mT).masked_fill_((near > rows) | (near <= rows - w), -math.inf),
                   (qt @ kd.mT).masked_fill_(far > rows - w, -math.inf)), -1)
    P = S.mul_(scale).softmax(-1)
    Pl, Pg = P[..., :k.shape[-2]], P[..., k.shape[-2]:]
    od = Pg @ vd
    return Pl @ v + od @ Uv, Pl, Pg, od


def _exact_sequence(case, s):
    """The causal forward, and for "train" its gradients, one batch element and block of rows at a time."""
    B, Hq, Hkv, N, w, dd = (case[n] for n in ("B", "Hq", "Hkv", "N", "w", "dd"))
    G, scale = Hq // Hkv, D_HEAD ** -0.5
    p = {n: t.double() for n, t in s.p.items()}
    grown = {n: t.repeat_interleave(G, 0) for n, t in p.items()}
    train = case["kind"] == "train"
    f64 = dict(dtype=torch.float64, device="cuda")
    out = torch.empty(s.q.shape, **f64)
    g = {n: torch.zeros(t.shape, **f64) for n, t in s.grads.items()} if train else {}
    step = max(64, min(N, int(3e8 / (Hq * N))))
    for b in range(B):
        k1, v1 = s.k[b].double(), s.v[b].double()
        kd1, vd1 = k1 @ p["Dk"], v1 @ p["Dv"]
        k, v, kd, vd = (t.repeat_interleave(G, 0) for t in (k1, v1, kd1, vd1))
        q = s.q[b].double()
        qt = s.qd[b].double() * (dd ** -0.5 / scale) if case.get("direct") else q @ grown["Uk"].mT
        if train:
            do = s.dout[b].double()
            dk, dv, dkd, dvd = (torch.zeros_like(t) for t in (k, v, kd, vd))
            dUk, dUv = torch.zeros_like(grown["Uk"]), torch.zeros_like(grown["Uv"])
        for r0 in range(0, N, step):
            r = slice(r0, min(N, r0 + step))
            a = slice(max(0, r0 - w + 1), r.stop)
            f = slice(0, max(0, r.stop - w))
            o, Pl, Pg, od = _attend(q[:, r], k[:, a], v[:, a], qt[:, r], kd[:, f], vd[:, f], grown["Uv"], r0, w,
                                    scale, a.start)
            out[b, :, r] = o
            if not train:
                continue
            d = do[:, r]
            dd_ = d @ grown["Uv"].mT
            row = (d * o).sum(-1, keepdim=True)
            dv[:, a] += Pl.mT @ d
            dvd[:, f] += Pg.mT @ dd_
            dUv += od.mT @ d
            dSl = Pl * ((d @ v[:, a].mT).sub_(row)).mul_(scale)
            dSg = Pg * ((dd_ @ vd[:, f].mT).sub_(row)).mul_(scale)
            dqt = dSg @ kd[:, f]
            g["dq"][b, :, r] = dSl @ k[:, a] + dqt @ grown["Uk"]
            dk[:, a] += dSl.mT @ q[:, r]
            dkd[:, f] += dSg.mT @ qt[:, r]
            dUk += dqt.mT @ q[:, r]
        if train:
            dk, dv, dkd, dvd, dUk, dUv = (t.view(Hkv, G, *t.shape[1:]).sum(1)
                                          for t in (dk, dv, dkd, dvd, dUk, dUv))
            g["dk"][b], g["dv"][b] = dk + dkd @ p["Dk"].mT, dv + dvd @ p["Dv"].mT
            g["dDk"] += k1.mT @ dkd
            g["dDv"] += v1.mT @ dvd
            g["dUk"] += dUk
            g["dUv"] += dUv
    return dict(out=out, **g) if train else out


def _exact_cached(case, s):
    """Cases on a cache: sequence by sequence, its keys and values gathered by position."""
    kind, w, Hkv = case["kind"], case["w"], case["Hkv"]
    c, before, new = s.cache, _lengths(case), _counts(case)
    latent = isinstance(c, dar.DarLatentCache)
    held = {n: (t.double() if t.is_floating_point() else t.clone()) for n, t in _held(c).items()}
    out = torch.zeros(s.out.shape, dtype=torch.float64, device="cuda") if hasattr(s, "out") else None
    table = c.block_table.long()
    scale = D_HEAD ** -0.5
    if latent:
        down = None
        if kind == "latent_decode":
            W_up, W_K, W_V = (t.double() for t in s.W)
            A_K, A_V = W_up @ W_K, W_up @ W_V
    else:
        p = {n: t.double() for n, t in s.p.items()}
        down = (p["Dk"], p["Dv"])
    for b, (L, n) in enumerate(zip(before, new)):
        near0 = max(0, L - w)  # the ring holds positions near0 .. L - 1
        slots = torch.arange(near0, L, device="cuda") % w
        kv = [t[b][:, slots].double() for t in (c.win_k, c.win_v)]
        if n:
            kv = [torch.cat((t, x[b, :, :n].double()), 1) for t, x in zip(kv, (s.k, s.v))]
        gone = max(0, L + n - w)  # positions below this one are out of the window after the call
        at = torch.arange(L if latent else near0, L + n if latent else gone, device="cuda")
        if len(at):
            page, r = table[b, at // PAGE], at % PAGE
            if latent:
                held["pool_c"][page, r] = s.h[b, :n].double() @ s.W_down.double()
            else:
                for name, x, W in zip(("pool_kd", "pool_vd"), kv, down):
                    held[name][page, :, r] = (x[:, :gone - near0] @ W).transpose(0, 1)
        if n:
            stay = torch.arange(max(L, gone), L + n, device="cuda")
            for name, x in zip(("win_k", "win_v"), kv):
                held[name][b][:, stay % w] = x[:, stay - near0]
            held["seq_lens"][b] = L + n
        if out is None:
            continue
        far = torch.arange(gone, device="cuda")
        G = case["Hq"] // Hkv
        if latent:
            cs = held["pool_c"][table[b, far // PAGE], far % PAGE]
            kd, vd, Uk, Uv = cs.expand(Hkv, -1, -1), cs.expand(Hkv, -1, -1), A_K, A_V
        else:
            page, r = table[b, far // PAGE], far % PAGE
            kd, vd = (held[m][page, :, r].transpose(0, 1) for m in ("pool_kd", "pool_vd"))
            Uk, Uv = p["Uk"], p["Uv"]
        q = s.q[b].double()
        q = q.view(Hkv, G, 1, D_HEAD) if kind != "chunk" else q.view(Hkv, G, n, D_HEAD)
        if case.get("direct"):
            qt = s.qd[b].double().view(Hkv, G, 1, case["dd"]) * (case["dd"] ** -0.5 / scale)
        else:
            qt = q @ Uk[:, None].mT
        o = _attend(q, kv[0][:, None], kv[1][:, None], qt, kd[:, None], vd[:, None], Uv[:, None],
                    L if kind == "chunk" else L + n - 1, w, scale, near0)[0]
        out[b] = o.reshape(out[b].shape)
    if kind in ("decode", "latent_decode"):
        return out
    return dict(held, out=out) if out is not None else held


def exact(case, seed):
    s = prepare(case, seed)
    return _exact_sequence(case, s) if case["kind"] in ("prefill", "train") else _exact_cached(case, s)
