"""The work that users of the attention path have it do, as cases that can be timed and checked.

A case is a dict of plain values; its ``kind`` names the entry point:

  train     ``mala.fwd`` and ``mala.bwd``: forward and backward of one self-attention call (training step)
  packed    ``mala.fwd_varlen`` and ``mala.bwd_varlen``: the same on packed sequences of different lengths
  prefill   ``mala.fwd_paged``: prefill chunks of several sequences behind prefixes that lie in a paged cache
  chunk     ``mala.fwd_chunk_split``: one chunk of new queries against a long context, keys cut into ranges
  decode    ``mala.decode`` / ``mala.decode_multi``: one or several new tokens over a contiguous bf16 cache
  dpaged    ``mala.decode_paged``: one or several new tokens over a paged bf16 cache, one length per sequence
  dfp8      ``mala.decode_fp8_paged``: one new token over a paged e4m3 cache

Inputs are the seeded workloads of ``workloads.py``: "literal" (heads that are diffuse, planted, peaked or look at
sinks; nearly every tile is retained), "R" (a quarter of the heads diffuse, the others sparse), "S" (every head sparse)
and, for decode, "D" (keys gated so that two thirds of the V tiles are retained).
"""
import math
import random

import torch

from paper_2609_32712_b200 import mala, workloads

TILE = 128


def listed():
    return [
        # one layer of a small model at a short context: latency of forward + backward (the 1K configuration)
        dict(name="train_1k_d64", kind="train", B=1, Hq=2, Hkv=2, N=1024, d=64, tau=1e-4, preset="literal"),
        # ordinary training context with full attention (tau = 0), grouped heads (the 8K configuration)
        dict(name="train_8k_full", kind="train", B=1, Hq=16, Hkv=4, N=8192, d=128, tau=0.0, preset="literal"),
        # long-context training on heads that retain nearly every tile (the 32K configuration, the headline)
        dict(name="train_32k", kind="train", B=1, Hq=32, Hkv=8, N=32768, d=128, tau=1e-4, preset="literal"),
        # one tensor-parallel rank's heads at 128K, most heads sparse (the 128K configuration's sizes)
        dict(name="train_128k_sparse", kind="train", B=1, Hq=8, Hkv=2, N=131072, d=128, tau=1e-4, preset="R"),
        # documents of ragged lengths packed into one training row
        dict(name="train_packed", kind="packed", Hq=16, Hkv=4, seqs=9, longest=6000, lens=11, d=128, tau=1e-4,
             preset="R"),
        # a serving batch of prefill chunks behind cached prefixes, pages of 64 keys
        dict(name="prefill_paged", kind="prefill", Hq=32, Hkv=8, seqs=8, chunk=2048, prefix=14000, lens=5, page=64,
             d=128, tau=1e-4, preset="R"),
        # the next chunk of one long prompt, heads of 256 columns
        dict(name="chunk_d256", kind="chunk", B=1, Hq=16, Hkv=4, Nq=1000, Nk=32768, d=256, splits=4, tau=1e-4,
             preset="R"),
        # long-context decode (the 128K decode configuration: 128 splits)
        dict(name="decode_128k", kind="decode", B=8, Hq=32, Hkv=8, Nk=131072, Sq=1, d=128, splits=128, tau=1e-4,
             preset="D"),
        # one short conversation: latency of a decode step
        dict(name="decode_single", kind="decode", B=1, Hq=32, Hkv=8, Nk=2000, Sq=1, d=128, splits=0, tau=1e-4,
             preset="literal"),
        # verification of four drafted tokens at a middle context
        dict(name="decode_verify4", kind="decode", B=4, Hq=32, Hkv=8, Nk=16389, Sq=4, d=128, splits=0, tau=1e-4,
             preset="D"),
        # a serving batch of conversations of different lengths, pages of 16 keys
        dict(name="decode_paged", kind="dpaged", B=32, Hq=32, Hkv=8, longest=16000, lens=7, page=16, Sq=1, d=128,
             tau=1e-4, preset="D"),
        # the same over an 8-bit cache, longer conversations, pages of 128 keys
        dict(name="decode_fp8", kind="dfp8", B=16, Hq=32, Hkv=8, longest=40000, lens=3, page=128, d=128, tau=1e-4,
             preset="D"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["train", "train", "packed", "prefill", "chunk", "decode", "decode", "dpaged", "dfp8"])
    tau = rng.choice([0.0, 1e-5, 1e-4, 1e-4, 1e-3])
    preset = rng.choice(["literal", "R", "R", "S"])
    heads = rng.choice([(2, 2), (8, 2), (16, 4), (32, 8)])
    c = dict(kind=kind, Hq=heads[0], Hkv=heads[1], tau=tau, preset=preset)
    if kind == "train":
        c.update(B=rng.choice([1, 1, 2]), N=_log(rng, 512, 32768), d=rng.choice([64, 96, 128, 128]))
        if c["N"] > 16384:
            c["B"] = 1
    elif kind == "packed":
        c.update(seqs=rng.randint(2, 12), longest=_log(rng, 300, 8000), lens=rng.randrange(1000),
                 d=rng.choice([64, 128, 128]))
    elif kind == "prefill":
        c.update(seqs=rng.randint(1, 12), chunk=_log(rng, 64, 4096), prefix=_log(rng, 128, 24000),
                 lens=rng.randrange(1000), page=rng.choice([16, 64, 128, 256]), d=rng.choice([64, 128, 128]))
    elif kind == "chunk":
        c.update(B=1, Nq=_log(rng, 64, 4096), Nk=_log(rng, 8192, 100000), d=rng.choice([128, 128, 256]),
                 splits=rng.choice([1, 2, 4, 8]))
        if c["d"] == 256:
            c.update(Hq=16, Hkv=4)
    else:
        c.update(B=_log(rng, 1, 32), preset=rng.choice(["literal", "D", "D"]))
        c.update(Hq=rng.choice([8, 32, 64]), Hkv=8)
        if kind == "decode":
            c.update(Nk=_log(rng, 500, 131072), Sq=rng.choice([1, 1, 1, 2, 4] if c["Hq"] < 64 else [1, 2]),
                     d=rng.choice([64, 128, 128, 256]), splits=0)
            if c["d"] == 256:
                c.update(Hq=16, Hkv=4)
            c["B"] = max(1, min(c["B"], (8 << 17) // c["Nk"]))
        else:
            c.update(longest=_log(rng, 500, 60000), lens=rng.randrange(1000), page=rng.choice([16, 64, 128, 256]), d=128)
            c["B"] = max(1, min(c["B"], (8 << 16) // c["longest"]))
            if kind == "dpaged":
                c.update(Sq=rng.choice([1, 1, 2]))
    return c


def _lens(n, longest, seed):
    """n lengths between a quarter of ``longest`` and all of it, the longest among them."""
    r = random.Random(seed)
    return [longest] + [r.randint(max(1, longest // 4), longest) for _ in range(n - 1)]


def _types(n):
    return [("diffuse", "sink", "peaked", "peaked")[h % 4] for h in range(n)]


def _head_types(c):
    return ["planted"] * c["Hq"] if c["Hq"] == 2 else _types(c["Hq"])


def _prefill(c, B, N, seed):
    return workloads.custom_prefill(B, c["Hq"], c["Hkv"], N, c["d"], head_types=_head_types(c), planted=8, seed=seed,
                                    preset=c["preset"], device="cuda")


def _decode(c, B, Nk, Sq, seed):
    """Queries [B,Sq,Hq,d] and caches; the queries of several new tokens are the newest one's with noise."""
    w = workloads.custom_decode(B, c["Hq"], c["Hkv"], Nk, c["d"], 1, group_types=_types(c["Hkv"]), seed=seed,
                                preset=c["preset"], device="cuda")
    if Sq > 1:
        g = torch.Generator(device="cuda")
        g.manual_seed(seed + 77)
        noise = torch.randn((B, Sq, c["Hq"], c["d"]), generator=g, device="cuda") * 0.5
        noise[..., -1] = 0.0                                      # the gate feature stays
        w["q"] = (w["q"].float() + noise).to(torch.bfloat16)
    return w


def _pool(x, page, seed):
    """Contiguous caches [B,N,...] (N a multiple of ``page``) as a shuffled pool of pages and its block table."""
    B, N = x.shape[:2]
    g = torch.Generator()
    g.manual_seed(seed)
    perm = torch.randperm(B * (N // page), generator=g).cuda()
    pages = torch.empty((B * (N // page), page) + tuple(x.shape[2:]), dtype=x.dtype, device=x.device)
    pages[perm] = x.reshape(pages.shape)
    return pages, perm.reshape(B, -1).to(torch.int32).contiguous()


def _i32(v):
    return torch.tensor(v, dtype=torch.int32, device="cuda")


def _cu(lens):
    out = [0]
    for n in lens:
        out.append(out[-1] + n)
    return out


def _chunk_lens(c):
    r = random.Random(c["lens"])
    nq = _lens(c["seqs"], c["chunk"], c["lens"])
    nk = [n + r.randint(0, c["prefix"]) for n in nq]
    nk[0] = nq[0] + c["prefix"]
    return nq, nk


def _ranges(c, B, Nk):
    """The split count of a decode step: the case's own, or the one that the library suggests."""
    return c.get("splits") or mala.decode_suggest_splits(B, c["Hkv"], Nk)


def _padded(n, page):
    return -(-n // page) * page


def prepare(c, seed):
    s = dict(c=c, scale=1.0 / math.sqrt(c["d"]), tau=c["tau"])
    kind = c["kind"]
    if kind == "train":
        w = _prefill(c, c["B"], c["N"], seed)
        s.update({x: w[x] for x in ("q", "k", "v", "do")})
    elif kind == "packed":
        lens = _lens(c["seqs"], c["longest"], c["lens"])
        w = workloads.pack_sequences([_prefill(c, 1, n, seed * 1000 + i) for i, n in enumerate(lens)])
        s.update({x: w[x] for x in ("q", "k", "v", "do")}, cu=w["cu_seqlens"], longest=max(lens))
    elif kind == "prefill":
        nq, nk = _chunk_lens(c)
        full = _padded(max(nk), max(c["page"], TILE))
        k = torch.zeros((c["seqs"], full, c["Hkv"], c["d"]), dtype=torch.bfloat16, device="cuda")
        v, q = torch.zeros_like(k), []
        for b in range(c["seqs"]):
            w = _prefill(c, 1, nk[b], seed * 1000 + b)
            k[b, :nk[b]], v[b, :nk[b]] = w["k"][0], w["v"][0]
            q.append(w["q"][0, nk[b] - nq[b]:])
        (kp, table), (vp, _) = _pool(k, c["page"], seed), _pool(v, c["page"], seed)
        s.update(q=torch.cat(q)[None].contiguous(), k=kp, v=vp, table=table, cu=_i32(_cu(nq)), seqlens=_i32(nk),
                 longest=max(nq))
    elif kind == "chunk":
        w = _prefill(c, c["B"], c["Nk"], seed)
        s.update(q=w["q"][:, c["Nk"] - c["Nq"]:].contiguous(), k=w["k"], v=w["v"])
        n = mala.workspace_bytes(mala.OP_FWD, c["B"], c["Hq"], c["Hkv"], c["Nq"], c["d"], c["splits"])
        s["ws"] = torch.empty(max(n, 256), dtype=torch.uint8, device="cuda")
    elif kind == "decode":
        w = _decode(c, c["B"], c["Nk"], c["Sq"], seed)
        s.update(q=w["q"], k=w["kcache"], v=w["vcache"], splits=_ranges(c, c["B"], c["Nk"]))
        n = mala.workspace_bytes(mala.OP_DECODE, c["B"] * c["Sq"], c["Hq"], c["Hkv"], c["Nk"], c["d"], s["splits"])
        s["ws"] = torch.empty(max(n, 256), dtype=torch.uint8, device="cuda")
    else:
        lens = _lens(c["B"], c["longest"], c["lens"])
        full, Sq = _padded(max(lens), max(c["page"], TILE)), c.get("Sq", 1)
        w = _decode(c, c["B"], full, Sq, seed)
        k, v = w["kcache"], w["vcache"]
        s.update(q=w["q"], seqlens=_i32(lens), splits=_ranges(c, c["B"], full))
        if kind == "dfp8":
            # one scale per 128-key tile, or per page where pages are smaller
            tile = min(c["page"], TILE)
            for x, t in (("k", k), ("v", v)):
                code, scales, _ = workloads.quantize_cache_e4m3(t, tile)
                s[x], s["table"] = _pool(code, c["page"], seed)
                per = scales.reshape(c["B"], c["Hkv"], full // c["page"], -1).permute(0, 2, 1, 3)
                s[x + "scale"] = _pool(per.contiguous(), 1, seed)[0][:, 0].contiguous()
        else:
            (s["k"], s["table"]), (s["v"], _) = _pool(k, c["page"], seed), _pool(v, c["page"], seed)
        n = mala.workspace_bytes(mala.OP_DECODE, c["B"] * Sq, c["Hq"], c["Hkv"], full, c["d"], s["splits"])
        s["ws"] = torch.empty(max(n, 256), dtype=torch.uint8, device="cuda")
    return s


def run(s):
    c, kind = s["c"], s["c"]["kind"]
    if kind == "train":
        qkv = (s["q"], s["k"], s["v"])
        o, lse, _ = mala.fwd(*qkv, s["scale"], s["tau"])
        dq, dk, dv, _ = mala.bwd(*qkv, o, s["do"], lse, s["scale"], s["tau"])
        return dict(o=o, lse=lse, dq=dq, dk=dk, dv=dv)
    if kind == "packed":
        qkv, seqs = (s["q"], s["k"], s["v"]), (s["cu"], s["longest"], s["scale"], s["tau"])
        o, lse, _ = mala.fwd_varlen(*qkv, *seqs)
        dq, dk, dv, _ = mala.bwd_varlen(*qkv, o, s["do"], lse, *seqs)
        return dict(o=o, lse=lse, dq=dq, dk=dk, dv=dv)
    if kind == "prefill":
        o, lse, _ = mala.fwd_paged(s["q"], s["k"], s["v"], s["cu"], s["table"], s["seqlens"], s["longest"], s["scale"],
                                   s["tau"])
    elif kind == "chunk":
        o, lse, _ = mala.fwd_chunk_split(s["q"], s["k"], s["v"], s["scale"], s["tau"], c["splits"], ws=s["ws"])
    elif kind == "decode":
        call = mala.decode if c["Sq"] == 1 else mala.decode_multi
        o, lse, _ = call(s["q"], s["k"], s["v"], s["scale"], s["tau"], s["splits"], ws=s["ws"])
    elif kind == "dpaged":
        o, lse, _ = mala.decode_paged(s["q"], s["k"], s["v"], s["table"], s["seqlens"], s["scale"], s["tau"], s["splits"],
                                      ws=s["ws"])
    else:
        o, lse, _ = mala.decode_fp8_paged(s["q"], s["k"], s["v"], s["kscale"], s["vscale"], s["table"], s["seqlens"],
                                          s["scale"], s["tau"], s["splits"], ws=s["ws"])
    return dict(o=o, lse=lse)


def _pairs(nq, nk):
    """Causal (query, key) pairs of the last nq of nk positions."""
    return nq * (nk - nq) + nq * (nq + 1) / 2


def work(c):
    """Bytes: every input read and every output written once.  Operations: every score (2 d per pair forward, and again
    in the backward) and, of the post-score work (2 d per pair forward, 8 d backward), all of it where nearly every
    tile is retained, and the share that belongs to the heads that are not sparse otherwise (the sparse heads' few
    retained tiles are left out: what has to be done there depends on the inputs)."""
    kind, Hq, Hkv, d, tau = c["kind"], c["Hq"], c["Hkv"], c["d"], c["tau"]
    share = 1.0
    if tau > 0 and c["preset"] in ("R", "S"):
        share = 0.0 if c["preset"] == "S" or Hq == 2 else 0.25
    row = 2 * d
    if kind in ("train", "packed"):
        shapes = [c["N"]] * c["B"] if kind == "train" else _lens(c["seqs"], c["longest"], c["lens"])
        rows, pairs = sum(shapes), Hq * sum(_pairs(n, n) for n in shapes)
        bytes_ = rows * row * (4 * Hq + 4 * Hkv)             # q, do, o, dq; k, v, dk, dv
        return dict(bytes=bytes_, flops=pairs * d * (4 + share * 10))
    if kind in ("prefill", "chunk"):
        nq, nk = _chunk_lens(c) if kind == "prefill" else ([c["Nq"]] * c["B"], [c["Nk"]] * c["B"])
        pairs = Hq * sum(_pairs(a, b) for a, b in zip(nq, nk))
        bytes_ = sum(nq) * Hq * (2 * row + 4) + sum(nk) * Hkv * row * (1 + share)
        return dict(bytes=bytes_, flops=pairs * d * (2 + share * 2))
    lens = [c["Nk"]] * c["B"] if kind == "decode" else _lens(c["B"], c["longest"], c["lens"])
    Sq, size = c.get("Sq", 1), 1 if kind == "dfp8" else 2
    # "D": the newest 128 keys and one tile in eight are live for three quarters of the KV heads
    vshare = 0.25 + 0.75 / 8 if tau > 0 and c["preset"] == "D" else 1.0
    return dict(bytes=sum(lens) * Hkv * d * size * (1 + vshare) + c["B"] * Sq * Hq * 4 * d,
                flops=sum(lens) * Sq * Hq * d * 2 * (1 + vshare))


def tolerance(c):
    # Probabilities, dS and the results are bf16.  Measured against 64 bits: outputs 0.9e-3 .. 2.4e-3, dV 2e-3, dQ and
    # dK (P and dS rounded, D from a rounded output) 6e-3 .. 7e-3; two correct results differ by up to twice that.
    return {"rel": 2e-2} if c["kind"] in ("train", "packed") else {"rel": 8e-3}


# ---- 64-bit results, by the definition (Eqs. 1-4 on 128 x 128 tiles) in plain torch ----

def _blocks(x, n, lead=0):
    """[N,H,d] as fp64 [H,n,128,d] with ``lead`` empty rows in front and zeros behind."""
    out = torch.zeros((n * TILE,) + tuple(x.shape[1:]), dtype=torch.float64, device=x.device)
    out[lead:lead + x.shape[0]] = x.double()
    return out.reshape(n, TILE, x.shape[1], x.shape[2]).permute(2, 0, 1, 3)


def _rows(xb, lead, n):
    return xb.permute(1, 2, 0, 3).reshape(-1, xb.shape[0], xb.shape[3])[lead:lead + n]


def _theta(tau, L):
    return torch.log(tau / L) if tau > 0 else torch.full_like(L, -math.inf)


def _positions(nq, nk, dev):
    """Query blocks by key position: first block, number of blocks, empty rows in the first, each padded row's position."""
    first, lead = (nk - nq) // TILE, (nk - nq) % TILE
    n = -(-(nq + lead) // TILE)
    pos = (first * TILE + torch.arange(n * TILE, device=dev)).reshape(n, TILE)
    return first, n, lead, pos, (pos >= nk - nq) & (pos < nk)


def _exact_fwd(q, k, v, scale, tau, splits=1):
    """(o, lse [Hq,Nq]) of the last Nq of Nk positions, keys in ``splits`` ranges."""
    (nq, Hq, d), (nk, Hkv, _) = q.shape, k.shape
    first, n, lead, pos, real = _positions(nq, nk, q.device)
    tk = -(-nk // TILE)
    qb = _blocks(q, n, lead).reshape(Hkv, Hq // Hkv, n, TILE, d)
    kb, vb = _blocks(k, tk), _blocks(v, tk)
    theta = _theta(tau, (pos + 1).double())
    per = -(-tk // splits)
    parts = []
    for r0 in range(0, tk, per):
        top = torch.clamp(first + torch.arange(n, device=q.device), max=min(r0 + per, tk) - 1)
        m = torch.full(qb.shape[:-1], -math.inf, dtype=torch.float64, device=q.device)
        l, o = torch.zeros_like(m), torch.zeros_like(qb)
        for t in range(int(top.max()) - r0 + 1):
            at = torch.nonzero(top - t >= r0)[:, 0]
            j = top[at] - t
            legal = (j[:, None] * TILE + torch.arange(TILE, device=q.device))[:, None, :] <= pos[at][:, :, None]
            s = (qb[:, :, at] @ kb[:, None, j].transpose(-1, -2)).mul_(scale).masked_fill_(~legal, -math.inf)
            top_s, m0, l0 = s.amax(-1), m[:, :, at], l[:, :, at]
            wants = (top_s > -math.inf) & ((l0 == 0) | (top_s - (m0 + torch.log(l0)) >= theta[at]))
            keep = (wants & real[at]).any(-1)[..., None]
            m1 = torch.where(keep, torch.maximum(m0, top_s), m0)
            ref = torch.where(m1 > -math.inf, m1, 0.0)
            p = s.sub_(ref[..., None]).exp_() * keep[..., None]
            f = torch.exp(m0 - ref)
            m[:, :, at], l[:, :, at] = m1, l0 * f + p.sum(-1)
            o[:, :, at] = o[:, :, at] * f[..., None] + p @ vb[:, None, j]
        parts.append((o / torch.where(l > 0, l, 1.0)[..., None], m + torch.log(l)))
    lse = torch.logsumexp(torch.stack([x[1] for x in parts]), 0)
    safe = torch.where(lse > -math.inf, lse, 0.0)
    o = sum(x[0] * torch.exp(x[1] - safe)[..., None] for x in parts)
    return _rows(o.reshape(Hq, n, TILE, d), lead, nq), lse.reshape(Hq, -1)[:, lead:lead + nq]


def _exact_bwd(q, k, v, o, lse, do, scale, tau):
    (n_, Hq, d), Hkv = q.shape, k.shape[1]
    n = -(-n_ // TILE)
    G = Hq // Hkv
    qb, dob, ob = (_blocks(x, n).reshape(Hkv, G, n, TILE, d) for x in (q, do, o))
    kb, vb = _blocks(k, n)[:, None], _blocks(v, n)[:, None]
    _, _, _, pos, real = _positions(n_, n_, q.device)
    lb = torch.full((Hq, n * TILE), math.inf, dtype=torch.float64, device=q.device)
    lb[:, :n_] = lse
    lb = lb.reshape(Hkv, G, n, TILE)
    theta, D = _theta(tau, (pos + 1).double()), (ob * dob).sum(-1)
    dq, dk, dv = torch.zeros_like(qb), torch.zeros_like(kb), torch.zeros_like(vb)
    for t in range(n):
        i, j = slice(t, n), slice(0, n - t)
        s = (qb[:, :, i] @ kb[:, :, j].transpose(-1, -2)).mul_(scale).sub_(lb[:, :, i, :, None])
        if t == 0:
            s = s.masked_fill_(pos[0][None, :] > pos[0][:, None], -math.inf)
        keep = (s.amax(-1) >= theta[i]).any(-1)[..., None, None]
        p = s.exp_() * keep
        ds = (dob[:, :, i] @ vb[:, :, j].transpose(-1, -2)).sub_(D[:, :, i, :, None]).mul_(p)
        dv[:, :, j] += (p.transpose(-1, -2) @ dob[:, :, i]).sum(1, keepdim=True)
        dk[:, :, j] += (ds.transpose(-1, -2) @ qb[:, :, i]).sum(1, keepdim=True)
        dq[:, :, i] += ds @ kb[:, :, j]
    shape = (Hq, n, TILE, d)
    return _rows(dq.reshape(shape), 0, n_) * scale, _rows(dk[:, 0], 0, n_) * scale, _rows(dv[:, 0], 0, n_)


def _exact_decode(q, k, v, nk, nmax, scale, tau, splits):
    """(o [Sq,Hq,d], lse [Sq,Hq]) of the last Sq of nk keys; splits laid out over nmax key positions."""
    (Sq, Hq, d), Hkv = q.shape, k.shape[1]
    per = -(-(-(-nmax // splits)) // TILE)                     # tiles of a split
    used = min(splits, -(-nk // (per * TILE)))
    kb, vb = (_blocks(x[:nk], used * per).reshape(Hkv, used, per, TILE, d) for x in (k, v))
    G = Hq // Hkv
    qb = q.double().reshape(Sq, Hkv, G, d).permute(1, 0, 2, 3).reshape(Hkv, 1, Sq * G, d)
    sees = (nk - Sq + 1 + torch.arange(Sq, device=q.device)).repeat_interleave(G)
    theta = _theta(tau, sees.clamp(min=1).double())
    m = torch.full((Hkv, used, Sq * G), -math.inf, dtype=torch.float64, device=q.device)
    l, o = torch.zeros_like(m), torch.zeros((Hkv, used, Sq * G, d), dtype=torch.float64, device=q.device)
    for t in range(per - 1, -1, -1):
        key = ((torch.arange(used, device=q.device) * per + t) * TILE)[:, None] + torch.arange(TILE, device=q.device)
        s = (qb @ kb[:, :, t].transpose(-1, -2) * scale).masked_fill(key[:, None, :] >= sees[:, None], -math.inf)
        top = s.amax(-1)
        keep = ((top > -math.inf) & ((l == 0) | (top - (m + torch.log(l)) >= theta))).any(-1)[..., None]
        m1 = torch.where(keep, torch.maximum(m, top), m)
        ref = torch.where(m1 > -math.inf, m1, 0.0)
        p, f = torch.exp(s - ref[..., None]) * keep[..., None], torch.exp(m - ref)
        m, l, o = m1, l * f + p.sum(-1), o * f[..., None] + p @ vb[:, :, t]
    ls = m + torch.log(l)
    lse = torch.logsumexp(ls, 1)
    out = (o / torch.where(l > 0, l, 1.0)[..., None] * torch.exp(ls - torch.where(lse > -math.inf, lse, 0.0)[:, None])[..., None]).sum(1)
    lay = lambda x: x.reshape(Hkv, Sq, G, -1).permute(1, 0, 2, 3).reshape(Sq, Hq, -1)  # noqa: E731
    return lay(out), lay(lse)[..., 0]


def _unpool(pages, table, n):
    return pages[table.long()].reshape((-1,) + tuple(pages.shape[2:]))[:n]


def exact(c, seed):
    s, kind = prepare(c, seed), c["kind"]
    scale, tau, split = s["scale"], s["tau"], c.get("splits", 1)
    with torch.no_grad():
        if kind in ("train", "packed"):
            if kind == "train":
                spans = [(b, 0, c["N"]) for b in range(c["B"])]
            else:
                cu = s["cu"].tolist()
                spans = [(0, cu[i], cu[i + 1]) for i in range(len(cu) - 1)]
            out = {x: torch.empty(s[y].shape, dtype=torch.float64, device="cuda")
                   for x, y in (("o", "q"), ("dq", "q"), ("dk", "k"), ("dv", "v"))}
            out["lse"] = torch.empty((len(s["q"]), c["Hq"], s["q"].shape[1]), dtype=torch.float64, device="cuda")
            for b, i, j in spans:
                q, k, v, do = (s[x][b, i:j] for x in ("q", "k", "v", "do"))
                o, lse = _exact_fwd(q, k, v, scale, tau)
                out["o"][b, i:j], out["lse"][b, :, i:j] = o, lse
                g = _exact_bwd(q, k, v, o, lse, do, scale, tau)
                out["dq"][b, i:j], out["dk"][b, i:j], out["dv"][b, i:j] = g
            if kind == "packed":
                out["lse"] = out["lse"][0]
            return out
        if kind == "prefill":
            nq, nk = _chunk_lens(c)
            cu, got = _cu(nq), []
            for b in range(c["seqs"]):
                k, v = (_unpool(s[x], s["table"][b], nk[b]) for x in ("k", "v"))
                got.append(_exact_fwd(s["q"][0, cu[b]:cu[b + 1]], k, v, scale, tau))
            return dict(o=torch.cat([x[0] for x in got])[None], lse=torch.cat([x[1] for x in got], 1))
        if kind == "chunk":
            got = [_exact_fwd(s["q"][b], s["k"][b], s["v"][b], scale, tau, split) for b in range(c["B"])]
            return dict(o=torch.stack([x[0] for x in got]), lse=torch.stack([x[1] for x in got]))
        got = []
        for b in range(c["B"]):
            if kind == "decode":
                k, v, nk, nmax = s["k"][b], s["v"][b], c["Nk"], c["Nk"]
            else:
                nk, nmax = int(s["seqlens"][b]), s["table"].shape[1] * c["page"]
                k, v = (_unpool(s[x], s["table"][b], nk) for x in ("k", "v"))
                if kind == "dfp8":
                    k, v = (x.view(torch.float8_e4m3fn).float().double() for x in (k, v))
                    tile = min(c["page"], TILE)
                    for x, y in ((k, "kscale"), (v, "vscale")):
                        per = s[y][s["table"][b].long()].permute(0, 2, 1).reshape(-1, c["Hkv"])
                        x *= per.double().repeat_interleave(tile, 0)[:nk, :, None]
            got.append(_exact_decode(s["q"][b], k, v, nk, nmax, scale, tau, s["splits"]))
        o, lse = torch.stack([x[0] for x in got]), torch.stack([x[1] for x in got])
        return dict(o=o, lse=lse[:, 0] if c.get("Sq", 1) == 1 else lse)
