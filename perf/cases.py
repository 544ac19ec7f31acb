"""The work that programs built on this library have it do, as timed cases.

Families (the "kind" of a case), each through its public entry points:
  step       one decode step: append the new K and V token, then attention over the packed cache
             (cobra_decode_step); "append": False is attention alone (cobra_decode_attn)
  rope       decode attention with the rotary embedding (cobra_decode_rope_attn)
  compress   a prefill's K and V into code rows (cobra_compress, one call per side)
  calibrate  calibration of many heads on the device (cobra_calibrate_heads)
  measure    measured distortion tables of many heads (cobra_measure_distortion)

Inputs.  Heads get power-law spectra and their (r, b) from the library's allocator at the case's
rate, an orthonormal basis each, and steps that fit the spectrum.  Rotated channels are near
Gaussian, so the codes that a cache holds are quantised normal numbers: a pool of code rows is
drawn per head and every cached row is a copy of one of them, which makes caches of gigabytes
quick to fill and lets exact() evaluate each distinct token once.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2609_24298_gb300 import cobra

D = 128
POOL_ROWS = 16  # distinct full code rows per head
DEV = "cuda"

# One layer's call of a model is the usual call of a serving engine: attention of a layer needs
# the output of the layer before it.  Calls over all layers are the shapes of the benchmark
# (replayed or batched layers), which the repository's workloads are quoted on.
LISTED = [
    # the smallest workload of the repository: one sequence, one layer, 2 bits per dimension;
    # latency and launches are what a user waits for
    dict(name="step_tiny", kind="step", append=True, layers=1, kv=8, group=4, seqs=1, tok_lo=2048, tok_hi=2048, bpd=2.0,
         joint=False, paged=False),
    # one layer of a chat server: a batch of short, ragged sequences in a paged cache
    dict(name="step_layer_chat", kind="step", append=True, layers=1, kv=8, group=4, seqs=24, tok_lo=131, tok_hi=6001,
         bpd=3.0, joint=False, paged=True),
    # one layer of the 8B-shaped model with long contexts at 1 bpd
    dict(name="step_layer_8b", kind="step", append=True, layers=1, kv=8, group=4, seqs=8, tok_lo=32768, tok_hi=32768,
         bpd=1.0, joint=False, paged=False),
    # the benchmark's step: all 32 layers of the 8B-shaped model, batch 8 x 32768 tokens, 1 bpd
    dict(name="step_model_8b", kind="step", append=True, layers=32, kv=8, group=4, seqs=8, tok_lo=32768, tok_hi=32768,
         bpd=1.0, joint=False, paged=False),
    # the 70B-shaped model: one 131072-token context, 8 query heads per kv head, K and V
    # allocated jointly at 0.5 bpd
    dict(name="step_model_70b", kind="step", append=True, layers=80, kv=8, group=8, seqs=1, tok_lo=131072,
         tok_hi=131072, bpd=0.5, joint=True, paged=False),
    # the ragged paged sweep at its highest rate (2 of the 32 layers, which are shaped alike)
    dict(name="step_ragged_4bpd", kind="step", append=True, layers=2, kv=8, group=4, seqs=32, tok_lo=1024, tok_hi=65536,
         bpd=4.0, joint=False, paged=True),
    # rotary decode: one layer, one sequence of an odd length
    dict(name="rope_layer", kind="rope", layers=1, kv=8, group=4, seqs=1, tok_lo=8191, tok_hi=8191, bpd=2.0, joint=False,
         paged=False),
    # rotary decode of the 8B-shaped cache (4 of the 32 layers)
    dict(name="rope_8b", kind="rope", layers=4, kv=8, group=4, seqs=8, tok_lo=32768, tok_hi=32768, bpd=1.0, joint=False,
         paged=False),
    # one layer's chunk of a chunked prefill, K and V, an odd number of tokens
    dict(name="compress_chunk", kind="compress", layers=1, kv=8, seqs=1, tokens=2001, bpd=4.0, paged=False),
    # the prefill benchmark: batch 64 x 4096 tokens at 4 bpd (8 of the 32 layers)
    dict(name="compress_prefill", kind="compress", layers=8, kv=8, seqs=64, tokens=4096, bpd=4.0, paged=False),
    # calibration of the K heads of the 8B-shaped model (attention-KL weights need the queries)
    dict(name="calibrate_8b_k", kind="calibrate", heads=256, tokens=512, queries=2048),
    # measured distortion tables of the same heads over the allocator's whole grid
    dict(name="measure_8b_k", kind="measure", heads=256, tokens=512, kl=True),
]

MAX_CODE_BYTES = 2 << 30  # packed bytes a drawn decode reads at most


def listed():
    return [dict(c) for c in LISTED]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_cache(rng, kind, max_bytes):
    c = dict(kind=kind)
    if kind == "step":
        c["append"] = rng.random() < 0.8
    c["layers"] = rng.choice([1, 1, 1, 2, 5, 16, 32])
    c["kv"] = rng.choice([1, 2, 4, 8, 8])
    c["group"] = rng.choice([4, 4, 8])
    c["seqs"] = _log_int(rng, 1, 64)
    hi = _log_int(rng, 17, 131072)
    c["tok_lo"], c["tok_hi"] = (hi, hi) if rng.random() < 0.5 else (max(1, hi // rng.randint(2, 50)), hi)
    c["bpd"] = rng.choice([0.5, 1.0, 1.5, 2.0, 3.0, 4.0])
    c["joint"] = rng.random() < 0.2
    c["paged"] = rng.random() < 0.5
    while _code_bytes(c) > max_bytes:
        if c["layers"] > 1:
            c["layers"] = max(1, c["layers"] // 2)
        elif c["seqs"] > 1:
            c["seqs"] = max(1, c["seqs"] // 2)
        else:
            c["tok_hi"] //= 2
            c["tok_lo"] = min(c["tok_lo"], c["tok_hi"])
    return c


def draw(rng):
    kind = rng.choice(["step", "step", "step", "rope", "compress", "compress", "calibrate", "measure"])
    if kind == "step":
        return _draw_cache(rng, kind, MAX_CODE_BYTES)
    if kind == "rope":
        return _draw_cache(rng, kind, MAX_CODE_BYTES // 8)
    if kind == "compress":
        c = dict(kind=kind, layers=rng.choice([1, 1, 2, 4]), kv=rng.choice([1, 2, 4, 8, 8]), seqs=_log_int(rng, 1, 64),
                 tokens=_log_int(rng, 1, 16384), bpd=rng.choice([0.5, 1.0, 2.0, 3.0, 4.0]), paged=rng.random() < 0.5)
        while c["layers"] * c["kv"] * c["seqs"] * c["tokens"] > 8 * 8 * 64 * 4096:
            c["seqs"] = max(1, c["seqs"] // 2)
        return c
    if kind == "calibrate":
        return dict(kind=kind, heads=_log_int(rng, 1, 256), tokens=rng.randint(160, 1024),
                    queries=rng.choice([0, rng.randint(100, 2048)]))
    return dict(kind=kind, heads=_log_int(rng, 1, 256), tokens=rng.randint(17, 512), kl=rng.random() < 0.5)


# ---------------------------------------------------------------------------------------
# heads
# ---------------------------------------------------------------------------------------
def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed((seed * 1000003 + stream * 7919 + 17) & 0x7FFFFFFFFFFFFFFF)
    return g


def _np_rng(seed, stream):
    return np.random.Generator(np.random.PCG64(np.random.SeedSequence([2609, seed, stream])))


def _spectra(rng, n, lo=0.3, hi=2.5):
    """Power-law eigenvalues i^-alpha, normalised to sum to 128 per head."""
    lam = np.arange(1, D + 1)[None, :] ** (-rng.uniform(lo, hi, n)[:, None])
    return lam * (D / lam.sum(axis=1, keepdims=True))


def _bases(n, gen):
    """n orthogonal 128 x 128 matrices (fp64): a sign-flipped Hadamard matrix reflected twice."""
    H = torch.ones((1, 1), dtype=torch.float64, device=DEV)
    while H.shape[0] < D:
        H = torch.cat([torch.cat([H, H], 1), torch.cat([H, -H], 1)], 0)
    s = torch.randint(0, 2, (n, 1, D), generator=gen, device=DEV).double() * 2 - 1
    M = (H / math.sqrt(D))[None] * s
    for _ in range(2):
        v = torch.randn((n, D, 1), generator=gen, device=DEV, dtype=torch.float64)
        v = v / v.norm(dim=1, keepdim=True)
        M = M - 2.0 * v @ (v.transpose(1, 2) @ M)
    return M


def _heads(n_side, bpd, joint, sides, seed):
    """(r, b, delta, W [n, 128, 128] fp32 with zero columns past r, mu [n, 128] fp32, sigma [n])."""
    rng = _np_rng(seed, 1)
    lam = _spectra(rng, sides * n_side)
    w = lam.copy()
    if not joint:  # K heads are weighted by the query energy along each direction
        w[:n_side] = -np.sort(-(lam[:n_side] * rng.permuted(_spectra(rng, n_side), axis=1)), axis=1)
    parts = [w] if joint else [w[i * n_side:(i + 1) * n_side] for i in range(sides)]
    res = [cobra.cobra_allocate(p, bpd) for p in parts]
    r, b = np.concatenate([x["r"] for x in res]), np.concatenate([x["b"] for x in res])
    L = np.array([0.0] + [cobra.cobra_loading_factor(k) for k in range(1, 9)])
    sigma = np.array([math.sqrt(lam[i, :r[i]].mean()) if r[i] else 0.0 for i in range(len(r))])
    delta = np.where(r > 0, 2.0 * L[b] * sigma / 2.0 ** b, 0.0).astype(np.float32)
    gen = _gen(seed, 2)
    W = _bases(len(r), gen).float()
    keep = torch.arange(D, device=DEV)[None, :] < torch.tensor(r, device=DEV)[:, None]
    W = W * keep[:, None, :]
    mu = (0.1 * torch.randn((len(r), D), generator=gen, device=DEV)).float()
    return r, b, delta, W, mu, sigma


def _cache_bytes(n_heads, bpd, n_slots):
    """Room for any allocation of n_heads heads at bpd: a program sizes its cache before it knows the heads."""
    return n_slots * 16 * int(bpd * D * n_heads) + 256 * n_heads


def _params(r, b, delta, W, mu, n_slots):
    """Parameter block of a set of heads and where each head's rows start in the cache."""
    offs, _ = cobra.cobra_plan_layout(r, b, n_slots)
    nbytes = cobra.cobra_params_bytes(r)
    block = torch.empty(nbytes, dtype=torch.uint8, device=DEV)
    Wh = W.cpu().numpy()
    cobra.cobra_params_build(block, nbytes, r, b, delta, offs, [Wh[i][:, :r[i]] for i in range(len(r))],
                             mu.cpu().numpy().reshape(-1))
    return block, offs


def _pack_rows(codes, r, b, side):
    """Code rows of the documented format: codes [..., 128 tokens, r] (int32) -> bytes [..., 16 r b]."""
    lead = codes.shape[:-2]
    c = codes.reshape(lead + (8, 2, 8, r // 2, 2))  # token = 16 tau + 8 u + p, channel = 2 s + i
    n = len(lead)
    ax = list(range(n))
    if side == 0:  # strip s, piece p, half i, rho = 2 tau + u
        c = c.permute(ax + [n + 3, n + 2, n + 4, n + 0, n + 1])
    else:  # p = 2 q + h: piece 4 i + q, half h
        c = c.reshape(lead + (8, 2, 4, 2, r // 2, 2))
        c = c.permute(ax + [n + 4, n + 5, n + 2, n + 3, n + 0, n + 1])
    c = c.reshape(lead + (r // 2, 8, 2, 16))
    words = torch.zeros(lead + (r // 2, 8, b, 2), dtype=torch.int32, device=codes.device)
    for rho in range(16):
        v, w, off = c[..., rho], (rho * b) >> 4, (rho * b) & 15
        words[..., w, :] |= (v << off) & 0xFFFF
        if off + b > 16:
            words[..., w + 1, :] |= v >> (16 - off)
    words = words[..., 0] | (words[..., 1] << 16)
    return words.contiguous().view(torch.uint8).reshape(lead + (16 * r * b,))


def _quantise(y, delta, b):
    """Codes of projected values, in 64 bits: y [..., r], delta and b plain numbers."""
    return torch.clamp(torch.floor(y.double() / float(delta) + 2.0 ** (b - 1)), 0, 2 ** b - 1).to(torch.int32)


# ---------------------------------------------------------------------------------------
# decode (step, rope)
# ---------------------------------------------------------------------------------------
def _lengths(case, seed):
    lo, hi, n = case["tok_lo"], case["tok_hi"], case["seqs"]
    T = _np_rng(seed, 3).integers(lo, hi + 1, size=n).astype(np.int64)
    T[0] = hi
    return T


def _cache_data(case, seed):
    """Everything about a decode's inputs but the buffers: heads, codes, lengths, tokens, queries."""
    L, H, G, S = case["layers"], case["kv"], case["group"], case["seqs"]
    n = L * H
    append = case["kind"] == "step" and case["append"]
    r, b, delta, W, mu, sigma = _heads(n, case["bpd"], case["joint"], 2, seed)
    T = _lengths(case, seed)
    rows = (T + 127) // 128
    gen = _gen(seed, 4)
    pool, last = [], []
    n_last = torch.tensor(T - 128 * (rows - 1), device=DEV)
    live = torch.arange(128, device=DEV)[None, :] < (n_last - (1 if append else 0))[:, None]  # [S, 128]
    for i in range(2 * n):
        ri, bi = int(r[i]), int(b[i])
        z = torch.randn((POOL_ROWS + S, 128, max(ri, 1)), generator=gen, device=DEV)[..., :ri]
        c = _quantise(z * float(sigma[i]), delta[i], bi) if ri else z.to(torch.int32)
        pool.append(c[:POOL_ROWS])
        last.append(c[POOL_ROWS:] * live[:, :, None])
    max_rows = int(rows.max())
    pick = torch.randint(0, POOL_ROWS, (2 * n, S, max_rows), generator=gen, device=DEV)
    # new tokens whose projections are distributed as the cached ones
    g = torch.randn((2 * n, S, D), generator=gen, device=DEV) * torch.tensor(sigma, device=DEV).float()[:, None, None]
    x = (mu[:, None, :] + g @ W.transpose(1, 2)).to(torch.bfloat16)  # [2n, S, 128]
    x = x.reshape(2, L, H, S, D).permute(0, 1, 3, 2, 4).contiguous()  # [side, L, S, H, 128]
    q = torch.randn((L, S, H * G, D), generator=gen, device=DEV).to(torch.bfloat16)
    return dict(r=r, b=b, delta=delta, W=W, mu=mu, T=T, rows=rows, pool=pool, last=last, pick=pick, x=x, q=q)


def _prepare_decode(case, seed):
    L, H, G, S = case["layers"], case["kv"], case["group"], case["seqs"]
    n = L * H
    d = _cache_data(case, seed)
    T, rows = d["T"], d["rows"]
    max_rows = int(rows.max())
    if case["paged"]:
        pages = (max_rows + 1) // 2
        n_slots = 2 * S * pages
        table = torch.tensor(_np_rng(seed, 5).permutation(S * pages).astype(np.int32).reshape(S, pages), device=DEV)
        rps, pps = 0, pages
    else:
        n_slots, table, rps, pps = S * max_rows, None, max_rows, 0
    block, offs = _params(d["r"], d["b"], d["delta"], d["W"], d["mu"], n_slots)
    cache = torch.zeros(_cache_bytes(2 * n, case["bpd"], n_slots), dtype=torch.uint8, device=DEV)
    # slot of (sequence, row) and which of the drawn rows it holds
    seq, row = np.concatenate([np.full(int(k), s) for s, k in enumerate(rows)]), np.concatenate([np.arange(int(k)) for k in rows])
    seq, row = torch.tensor(seq, device=DEV), torch.tensor(row, device=DEV)
    is_last = row == torch.tensor(rows, device=DEV)[seq] - 1
    slot = seq * max_rows + row if table is None else 2 * table[seq, row // 2].long() + row % 2
    for i in range(2 * n):
        ri, bi = int(d["r"][i]), int(d["b"][i])
        if not ri:
            continue
        packed = _pack_rows(torch.cat([d["pool"][i], d["last"][i]]), ri, bi, i // n)
        src = torch.where(is_last, POOL_ROWS + seq, d["pick"][i][seq, row])
        region = cache[int(offs[i]):int(offs[i]) + n_slots * packed.shape[1]].view(n_slots, packed.shape[1])
        region[slot] = packed[src]
    q_stride = dict(q_stride_layer=S * H * G * D, q_stride_seq=H * G * D, o_stride_layer=S * H * G * D, o_stride_seq=H * G * D)
    desc = cobra.decode_desc(k_head0=0, v_head0=n, layer_stride=H, n_layers=L, n_kv_heads=H, group=G, n_seqs=S,
                             rows_per_seq=rps, pages_per_seq=pps, **q_stride)
    cap = T.astype(np.int32)
    hb = np.where(d["r"] > 0, d["b"], 0)
    ws_bytes = cobra.cobra_decode_workspace_size(desc, d["r"], hb, cap)
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device=DEV)
    info = cobra.cobra_decode_plan(desc, d["r"], hb, cap, ws, ws_bytes)
    st = dict(case=case, block=block, cache=cache, desc=desc, ws=ws, ws_bytes=ws_bytes, info=info, table=table, q=d["q"],
              lens=torch.tensor(cap, device=DEV), out=torch.zeros((L, S, H * G, D), dtype=torch.float32, device=DEV))
    if case["kind"] == "step":
        side = lambda s: cobra.compress_desc(head0=s * n, layer_stride=H, n_layers=L, n_kv_heads=H, side=s, n_seqs=S,
                                             rows_per_seq=rps, pages_per_seq=pps, x_stride_layer=S * H * D,
                                             x_stride_seq=H * D, x_stride_tok=H * D, x_stride_head=D)
        st.update(kdesc=side(0), vdesc=side(1), k_new=d["x"][0].contiguous(), v_new=d["x"][1].contiguous(),
                  pos=torch.tensor(cap - 1, device=DEV))
    else:
        st["max_pos"] = int(T.max())
        nbytes = cobra.cobra_rope_table_bytes(st["max_pos"])
        st["rope"] = torch.empty(nbytes // 4, dtype=torch.float32, device=DEV)
        cobra.cobra_rope_table(500000.0, st["max_pos"], st["rope"], nbytes)
    return st


def _run_decode(s):
    if s["case"]["kind"] == "rope":
        cobra.cobra_decode_rope_attn(s["block"], s["desc"], s["info"], s["q"], None, s["rope"], s["max_pos"], s["cache"],
                                     s["lens"], s["table"], s["out"], s["ws"], s["ws_bytes"])
        return {"out": s["out"]}
    if not s["case"]["append"]:
        cobra.cobra_decode_attn(s["block"], s["desc"], s["info"], s["q"], s["cache"], s["lens"], s["table"], s["out"],
                                s["ws"], s["ws_bytes"])
        return {"out": s["out"]}
    cobra.cobra_decode_step(s["block"], s["desc"], s["info"], s["kdesc"], s["vdesc"], s["k_new"], s["v_new"], s["pos"],
                            s["q"], s["cache"], s["lens"], s["table"], s["out"], s["ws"], s["ws_bytes"])
    return {"out": s["out"], "cache": s["cache"]}


def _rotate(x, angle):
    """The rotate-half form: pairs (j, j + 64) of x [..., 128] turned by angle [..., 64]."""
    c, s, a, b = torch.cos(angle), torch.sin(angle), x[..., :64], x[..., 64:]
    return torch.cat([a * c - b * s, a * s + b * c], dim=-1)


def _exact_decode(case, seed):
    """Attention over the dequantised cache in 64 bits.  Without the rotary embedding a token's
    score depends on its codes alone, so each pool token is scored once and weighted by how often
    the sequence holds it."""
    L, H, G, S = case["layers"], case["kv"], case["group"], case["seqs"]
    n = L * H
    rope = case["kind"] == "rope"
    append = case["kind"] == "step" and case["append"]
    d = _cache_data(case, seed)
    T, rows = d["T"], d["rows"]
    omega = 500000.0 ** (-2.0 * torch.arange(64, device=DEV, dtype=torch.float64) / D)
    out = torch.zeros((L, S, H * G, D), dtype=torch.float64, device=DEV)

    def values(i, codes):  # dequantised, rotated back
        ri = int(d["r"][i])
        z = float(d["delta"][i]) * (codes.double() - 2.0 ** (int(d["b"][i]) - 1) + 0.5)
        return d["mu"][i].double() + z @ d["W"][i].double()[:, :ri].T

    for i in range(n):
        l, h = divmod(i, H)
        side = []
        for s, j in ((0, i), (1, n + i)):
            last = d["last"][j].clone()
            if append:
                y = (d["x"][s, l, :, h].double() - d["mu"][j].double()) @ d["W"][j].double()[:, :int(d["r"][j])]
                if y.shape[1]:
                    at = torch.tensor((T - 1) % 128, device=DEV)
                    last[torch.arange(S, device=DEV), at] = _quantise(y, d["delta"][j], int(d["b"][j]))
            side.append((values(j, d["pool"][j].reshape(POOL_ROWS * 128, -1)), values(j, last)))
        (kp, kl), (vp, vl) = side
        for s in range(S):
            Ts, R = int(T[s]), int(rows[s])
            q = d["q"][l, s, h * G:(h + 1) * G].double() / math.sqrt(D)
            rest = Ts - 128 * (R - 1)
            pk, pv = d["pick"][i, s, :R - 1], d["pick"][n + i, s, :R - 1]
            if rope:
                k = torch.cat([kp.view(POOL_ROWS, 128, D)[pk].reshape(-1, D), kl[s, :rest]])
                v = torch.cat([vp.view(POOL_ROWS, 128, D)[pv].reshape(-1, D), vl[s, :rest]])
                pos = torch.arange(Ts, device=DEV, dtype=torch.float64)
                k = _rotate(k, pos[:, None] * omega)
                q = _rotate(q, (Ts - 1) * omega)
                out[l, s, h * G:(h + 1) * G] = torch.softmax(q @ k.T, dim=1) @ v
            else:
                sc = (q @ kp.T).view(G, POOL_ROWS, 128)[:, pk].reshape(G, -1)  # scores of the full rows' tokens
                sc = torch.cat([sc, q @ kl[s, :rest].T], dim=1)
                p = torch.softmax(sc, dim=1)
                wv = torch.zeros((G, POOL_ROWS, 128), dtype=torch.float64, device=DEV)
                wv.index_add_(1, pv, p[:, :128 * (R - 1)].reshape(G, R - 1, 128))
                out[l, s, h * G:(h + 1) * G] = wv.reshape(G, -1) @ vp + p[:, 128 * (R - 1):] @ vl[s, :rest]
    res = {"out": out}
    if append:
        res["cache"] = None  # bytes
    return res


def _mean_len(case):
    return case["tok_hi"] if case["tok_lo"] == case["tok_hi"] else 0.5 * (case["tok_lo"] + case["tok_hi"])


def _code_bytes(case):
    return 2 * case["layers"] * case["kv"] * case["seqs"] * _mean_len(case) * D * case["bpd"] / 8


def _work_decode(case):
    # a rank of about 64 stands for the allocator's mix
    L, H, G, S, r = case["layers"], case["kv"], case["group"], case["seqs"], 64
    heads, toks = L * H, L * H * S * _mean_len(case)
    small = heads * (2 * r * D * 4) + heads * S * G * D * (2 + 4) + heads * S * 2 * D * 2
    flops = toks * 4 * r * G
    if case["kind"] == "rope":
        flops = toks * (2 * D * r + 2 * D * G + 2 * r * G)
    return {"bytes": _code_bytes(case) + small, "flops": flops}


# ---------------------------------------------------------------------------------------
# compress
# ---------------------------------------------------------------------------------------
def _compress_data(case, seed):
    L, H, S, T = case["layers"], case["kv"], case["seqs"], case["tokens"]
    r, b, delta, W, mu, sigma = _heads(L * H, case["bpd"], False, 2, seed)
    rng, gen = _np_rng(seed, 6), _gen(seed, 7)
    scale = np.ones((2, L, H, D), np.float32)
    for idx in np.ndindex(2, L, H):  # four outlier coordinates per head
        scale[idx][rng.choice(D, 4, replace=False)] = 8.0
    # the bases mix all coordinates, so every projected channel has about the mean variance
    rms = math.sqrt((D - 4 + 4 * 64.0) / D)
    sig = np.where(sigma > 0, sigma, 1.0).reshape(2, L, H, 1)
    scale = torch.tensor((scale / rms * sig).astype(np.float32), device=DEV)
    x = []
    for side in range(2):
        t = torch.empty((L, S, T, H, D), dtype=torch.bfloat16, device=DEV)
        m = mu.view(2, L, H, D)[side]
        for l in range(L):
            g = torch.randn((S, T, H, D), generator=gen, device=DEV)
            t[l] = g.mul_(scale[side, l]).add_(m[l])
        x.append(t)
    return r, b, delta, W, mu, sigma, x


def _prepare_compress(case, seed):
    L, H, S, T = case["layers"], case["kv"], case["seqs"], case["tokens"]
    r, b, delta, W, mu, sigma, x = _compress_data(case, seed)
    rows = (T + 127) // 128
    pages = (rows + 1) // 2
    table = None
    if case["paged"]:
        table = torch.tensor(_np_rng(seed, 5).permutation(S * pages).astype(np.int32).reshape(S, pages), device=DEV)
    n_slots = 2 * S * pages if case["paged"] else S * rows
    block, offs = _params(r, b, delta, W, mu, n_slots)
    cache = torch.zeros(_cache_bytes(2 * L * H, case["bpd"], n_slots), dtype=torch.uint8, device=DEV)
    descs = [cobra.compress_desc(head0=s * L * H, layer_stride=H, n_layers=L, n_kv_heads=H, side=s, n_seqs=S,
                                 rows_per_seq=0 if case["paged"] else rows, pages_per_seq=pages if case["paged"] else 0,
                                 x_stride_layer=S * T * H * D, x_stride_seq=T * H * D, x_stride_tok=H * D, x_stride_head=D)
             for s in range(2)]
    return dict(case=case, block=block, cache=cache, table=table, descs=descs, x=x, offs=offs, r=r, b=b)


def _run_compress(s):
    for side in range(2):
        cobra.cobra_compress(s["block"], s["descs"][side], s["x"][side], 0, s["case"]["tokens"], s["cache"], s["table"])
    return s["cache"]


def _exact_compress(case, seed):
    """The code rows from a projection in 64 bits (bytes: codes at a cell boundary may differ)."""
    L, H, S, T = case["layers"], case["kv"], case["seqs"], case["tokens"]
    if L * H * S * T > 1 << 22:
        return None  # the 64-bit projections take too long
    r, b, delta, W, mu, sigma, x = _compress_data(case, seed)
    rows = (T + 127) // 128
    pages = (rows + 1) // 2
    n_slots = 2 * S * pages if case["paged"] else S * rows
    offs, _ = cobra.cobra_plan_layout(r, b, n_slots)
    cache = torch.zeros(_cache_bytes(2 * L * H, case["bpd"], n_slots), dtype=torch.uint8, device=DEV)
    slot = torch.arange(S * rows, device=DEV)
    if case["paged"]:
        table = torch.tensor(_np_rng(seed, 5).permutation(S * pages).reshape(S, pages), device=DEV)
        row = torch.arange(rows, device=DEV)
        slot = (2 * table[:, row // 2] + row % 2).reshape(-1)
    for i in range(2 * L * H):
        ri, bi = int(r[i]), int(b[i])
        if not ri:
            continue
        side, l, h = i // (L * H), (i // H) % L, i % H
        y = (x[side][l, :, :, h].double() - mu[i].double()) @ W[i].double()[:, :ri]
        c = torch.zeros((S, rows * 128, ri), dtype=torch.int32, device=DEV)
        c[:, :T] = _quantise(y, delta[i], bi)
        packed = _pack_rows(c.view(S * rows, 128, ri), ri, bi, side)
        region = cache[int(offs[i]):int(offs[i]) + n_slots * packed.shape[1]].view(n_slots, packed.shape[1])
        region[slot] = packed
    return cache


def _work_compress(case):
    tok = 2 * case["layers"] * case["kv"] * case["seqs"] * case["tokens"]
    r = min(D, 64 * max(1.0, case["bpd"] / 2))  # about the mean rank of the allocator's mix
    return {"bytes": tok * (2 * D + D * case["bpd"] / 8) + 2 * case["layers"] * case["kv"] * D * r * 4,
            "flops": tok * 2 * D * r}


# ---------------------------------------------------------------------------------------
# calibration and measured distortion
# ---------------------------------------------------------------------------------------
def _tokens(n, count, seed, stream, lo=0.3, hi=2.5):
    """[n, count, 128] fp32 vectors (bf16 values) x = S R diag(sqrt(lambda)) g, four coordinates x 8."""
    rng, gen = _np_rng(seed, stream), _gen(seed, stream)
    lam = torch.tensor(_spectra(rng, n, lo, hi), device=DEV)
    scale = np.ones((n, D, 1))
    for i in range(n):
        scale[i, rng.choice(D, 4, replace=False)] = 8.0
    A = torch.tensor(scale, device=DEV) * _bases(n, gen) * lam.sqrt()[:, None, :]
    x = torch.randn((n, count, D), generator=gen, device=DEV) @ A.float().transpose(1, 2)
    x = x + 0.3 * torch.randn((n, 1, D), generator=gen, device=DEV)
    return x.to(torch.bfloat16).float().contiguous()


def _calib_inputs(case, seed):
    x = _tokens(case["heads"], case["tokens"], seed, 10)
    q = _tokens(case["heads"], case["queries"], seed, 11) if case["queries"] else None
    return x, q


def _prepare_calibrate(case, seed):
    n = case["heads"]
    x, q = _calib_inputs(case, seed)
    f64 = lambda *s: torch.zeros(s, dtype=torch.float64, device=DEV)
    return dict(case=case, x=x, q=q, mu=f64(n, D), lam=f64(n, D), U=f64(n, D * D), w=f64(n, D))


def _run_calibrate(s):
    cobra.cobra_calibrate_heads(s["x"], s["q"], s["mu"], s["lam"], s["U"], s["w"])
    return {k: s[k] for k in ("mu", "lam", "U", "w")}


def _eigen(x, q):
    """(mu, lam, U with directions as rows, w) in the allocator's order, 64 bits."""
    x = x.double()
    mu = x.mean(dim=1)
    xc = x - mu[:, None, :]
    lam, V = torch.linalg.eigh((xc.transpose(1, 2) @ xc / x.shape[1]).cpu())
    lam, V = lam.flip(1).to(DEV), V.flip(2).transpose(1, 2).to(DEV)  # descending, directions as rows
    big = V.gather(2, V.abs().argmax(dim=2, keepdim=True))
    V = V * torch.where(big < 0, -1.0, 1.0)
    w = lam.clone()
    if q is not None:
        w = ((V @ q.double().transpose(1, 2)) ** 2).mean(dim=2) * lam
        order = torch.sort(-w, dim=1, stable=True).indices
        lam, w = lam.gather(1, order), w.gather(1, order)
        V = V.gather(1, order[:, :, None].expand_as(V))
    return mu, lam, V, w


def _exact_calibrate(case, seed):
    mu, lam, V, w = _eigen(*_calib_inputs(case, seed))
    return {"mu": mu, "lam": lam, "U": V.reshape(case["heads"], -1), "w": w}


def _work_calibrate(case):
    n, t, q = case["heads"], case["tokens"], case["queries"]
    # moments of tokens and queries (upper triangles), reduction to tridiagonal form, its
    # eigenvectors and their transformation back, the variances along the directions
    flops = n * (t * D * (D + 1) + q * D * (D + 1) + (4 / 3 + 3 + 2) * D ** 3 + (2 * D ** 3 if q else 0))
    return {"bytes": n * (4 * D * (t + q) + 8 * (D * D + 3 * D)), "flops": flops}


RANKS, BITS = list(range(0, D + 1, 2)), list(range(1, 9))


def _measure_inputs(case, seed):
    n = case["heads"]
    rng, gen = _np_rng(seed, 12), _gen(seed, 12)
    # a calibration's results: eigenvalues and weights, directions in descending order of weight
    lam = _spectra(rng, n)
    w = lam * rng.permuted(_spectra(rng, n), axis=1) if case["kl"] else lam
    order = np.argsort(-w, axis=1, kind="stable")
    lam = torch.tensor(np.take_along_axis(lam, order, axis=1), device=DEV)
    w = torch.tensor(np.take_along_axis(w, order, axis=1), device=DEV)
    U = _bases(n, gen).float()  # direction k = row k
    c = torch.randn((n, case["tokens"], D), generator=gen, device=DEV) * lam.sqrt().float()[:, None, :]
    mu = 0.3 * torch.randn((n, D), generator=gen, device=DEV)
    x = (mu[:, None, :] + c @ U).to(torch.bfloat16).float().contiguous()
    signs = (torch.randint(0, 2, (n, D), generator=gen, device=DEV) * 2 - 1).to(torch.int8)
    return x, U.reshape(n, D * D).contiguous(), lam, w, mu, signs


def _prepare_measure(case, seed):
    n = case["heads"]
    x, U, lam, w, mu, signs = _measure_inputs(case, seed)
    return dict(case=case, x=x, U=U, lam=lam, w=w, mu=mu, signs=signs,
                coords=torch.empty((n, case["tokens"], D), dtype=torch.float32, device=DEV),
                D=torch.zeros((n, len(RANKS), len(BITS)), dtype=torch.float64, device=DEV))


def _run_measure(s):
    cobra.cobra_measure_distortion(s["x"], s["U"], s["lam"], s["w"], s["mu"], s["signs"], RANKS, BITS, s["coords"], s["D"])
    return s["D"]


def _loading(b):
    """The loading factor of the 2^b-cell quantiser, a constant per width (a setting, not a result)."""
    return cobra.cobra_loading_factor(b)


def _block_hadamard(r):
    """Block-diagonal normalised Sylvester matrices of the binary digits of r, largest first."""
    H, o = torch.zeros((r, r), dtype=torch.float64, device=DEV), 0
    for p in range(7, -1, -1):
        if r >> p & 1:
            B = torch.ones((1, 1), dtype=torch.float64, device=DEV)
            for _ in range(p):
                B = torch.cat([torch.cat([B, B], 1), torch.cat([B, -B], 1)], 0)
            H[o:o + 2 ** p, o:o + 2 ** p] = B / math.sqrt(2 ** p)
            o += 2 ** p
    return H


def _exact_measure(case, seed):
    x, U, lam, w, mu, signs = _measure_inputs(case, seed)
    n = case["heads"]
    omega = torch.where(lam > 0, w / lam, torch.zeros_like(w))
    c = (x.double() - mu.double()[:, None]) @ U.double().view(n, D, D).transpose(1, 2)
    out = torch.zeros((n, len(RANKS), len(BITS)), dtype=torch.float64, device=DEV)
    for i, r in enumerate(RANKS):
        tail = (c[:, :, r:] ** 2 * omega[:, None, r:]).sum(dim=2).mean(dim=1)
        H = _block_hadamard(r)[None] * signs[:, None, :r].double()  # [n, r, r]
        y = c[:, :, :r] @ H.transpose(1, 2)
        for j, b in enumerate(BITS):
            out[:, i, j] = tail
            if r:
                delta = (2.0 * _loading(b) * lam[:, :r].mean(dim=1).sqrt() / 2 ** b).float().double()[:, None, None]
                code = torch.clamp(torch.floor(y / delta + 2.0 ** (b - 1)), 0, 2 ** b - 1)
                e = (y - delta * (code - 2.0 ** (b - 1) + 0.5)) @ H
                out[:, i, j] += (e * e * omega[:, None, :r]).sum(dim=2).mean(dim=1)
    return out


def _work_measure(case):
    n, t = case["heads"], case["tokens"]
    # per kept coordinate and width: quantise and accumulate, with KL weights also turned back
    per = len(BITS) * (8 + (8 if case["kl"] else 0))
    return {"bytes": n * (4 * D * t + 4 * D * D + 8 * len(RANKS) * len(BITS)),
            "flops": n * t * (2 * D * D + sum(RANKS) * per)}


# ---------------------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("step", "rope"):
        return _prepare_decode(case, seed)
    return {"compress": _prepare_compress, "calibrate": _prepare_calibrate, "measure": _prepare_measure}[kind](case, seed)


def run(state):
    kind = state["case"]["kind"]
    if kind in ("step", "rope"):
        return _run_decode(state)
    return {"compress": _run_compress, "calibrate": _run_calibrate, "measure": _run_measure}[kind](state)


def work(case):
    kind = case["kind"]
    if kind in ("step", "rope"):
        return _work_decode(case)
    return {"compress": _work_compress, "calibrate": _work_calibrate, "measure": _work_measure}[kind](case)


def tolerance(case):
    kind = case["kind"]
    if kind in ("step", "rope"):
        # probabilities are rounded to fp16 (2^-12 each) before the value sums: 2e-5 to 1.4e-4
        # against 64 bits; a code of the new token at a cell boundary may fall on either side
        return {"rel": 6e-4, "max": 1e-2, "differ": 1e-5}
    if kind == "compress":
        # a code whose value lies within 1e-4 of a cell boundary may fall on either side
        return {"differ": 1e-4}
    if kind == "calibrate":
        # 64-bit results; a direction's error grows with the inverse of its eigenvalue's gap
        # (6e-11 over all directions against LAPACK)
        return {"rel": 1e-9, "max": 1e-5}
    # fp32 sums over tokens, single codes at a cell boundary: 1e-5 to 3e-5 against 64 bits
    return {"rel": 1.3e-4, "max": 5e-3}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("step", "rope"):
        return _exact_decode(case, seed)
    return {"compress": _exact_compress, "calibrate": _exact_calibrate, "measure": _exact_measure}[kind](case, seed)
