"""The workloads whose speed this library is judged by, each one a call (or a
short sequence of calls) that a recurrent-depth model makes at a step.

Shapes and selection rules are those of the benchmark workloads (tiny, 4K, 4K
batched with 55 heads of 96, 16K, 32K with grouped queries, 4K at block 32)
and ragged lengths between them.  Inputs follow the recipe of those workloads
on the GPU: normal Q, K, V, key blocks with a signature that the query blocks
they are planted in pull towards, a geometric drift between recurrent steps.
Supports are lists of the form a selection produces: sink, local window,
planted blocks, and further blocks up to the cap.
"""
import math

import torch

from paper_2609_27373_gb300 import wise

DEV = "cuda"

# kind: late      one late step, wise_sparse_attn
#       dense     one unrestricted step, wise_full_attn_accumulate without mass
#       discover  two discovery steps, wise_full_attn_accumulate with mass
#       select    wise_select_support from accumulated mass
#       diagnose  working set of four steps, retained mass, overlap with the running support
#       frozen    one late step from a stored distribution, wise_frozen_pv


def _attn(name, kind, b, L, h, hkv, d, blk, cap=0, sink=1, local=1, planted=3, boost=2.5, std=1.0):
    return {"name": name, "kind": kind, "batch": b, "seqlen": L, "heads": h, "kv_heads": hkv, "dim": d, "block": blk,
            "cap": cap, "sink": sink, "local": local, "planted": planted, "boost": boost, "std": std}


def listed():
    return [
        # The smallest late step: a short context, four heads; launch and latency count.
        _attn("late_tiny", "late", 1, 512, 4, 4, 64, 64, cap=4, planted=2, boost=3.0, std=0.125),
        # The ordinary late step: 28 of the 32 recurrent steps of a 4K trajectory are this call.
        _attn("late_4k", "late", 1, 4096, 32, 32, 128, 128, cap=8),
        # The same at the paper's block of 32 keys, with the same key budget per query block.
        _attn("late_4k_b32", "late", 1, 4096, 32, 32, 128, 32, cap=32),
        # Batched requests, the paper's 55 heads of 96.
        _attn("late_4k_b4_d96", "late", 4, 4096, 55, 55, 96, 128, cap=8, planted=4, boost=3.0),
        # Long context: 16K, window of two blocks.
        _attn("late_16k", "late", 1, 16384, 32, 32, 128, 128, cap=11, local=2, planted=4, boost=3.0),
        # The longest: 32K with four query heads to a kv head.
        _attn("late_32k_gqa", "late", 1, 32768, 32, 8, 128, 128, cap=15, local=2, planted=6, boost=3.0),
        # Two of the discovery steps that open a 4K trajectory (the first writes the mass, the second adds to it).
        _attn("discover_4k", "discover", 1, 4096, 32, 32, 128, 128),
        # A discovery on a ragged length with grouped queries, heads of 64 and small blocks.
        _attn("discover_1952_b32", "discover", 1, 1952, 12, 4, 64, 32),
        # A step without mass: the full attention that late steps are compared with, or a layer kept dense.
        _attn("dense_4k", "dense", 1, 4096, 32, 32, 128, 128),
        # The selection at the end of the discovery, at the longest context.
        _attn("select_32k", "select", 1, 32768, 32, 8, 128, 128, cap=15, local=2, planted=6),
        # Routing diagnostics of a 4K trajectory: the union working set of four steps, the mass that the running
        # support retains, its overlap with the working set.
        _attn("diagnose_4k", "diagnose", 1, 4096, 32, 32, 128, 128, cap=8),
        # Freeze-A from a stored distribution: one late step.
        _attn("frozen_4k", "frozen", 1, 4096, 32, 32, 128, 128, cap=8),
    ]


def draw(rng):
    """A case of the same ranges: the kinds above, lengths 256 .. 32768 (multiples of the block, most of them
    ragged against the 128-row tiles at block 32 and 64), heads and batch so that the work stays below that of
    the largest listed case of its kind."""
    kind = rng.choice(["late", "late", "late", "late", "discover", "discover", "dense", "select", "diagnose", "frozen"])
    d = rng.choice([64, 96, 128, 128])
    blk = 128 if kind == "frozen" else rng.choice([32, 64, 128, 128])
    top = {"late": 32768, "dense": 8192, "discover": 8192, "select": 32768, "diagnose": 8192, "frozen": 8192}[kind]
    if blk == 32 and kind in ("select", "late"):
        top = 16384
    L = blk * max(1, round(math.exp(rng.uniform(math.log(256), math.log(top))) / blk))
    nb = L // blk
    group = rng.choice([1, 1, 2, 3, 4, 8])
    b = rng.choice([1, 1, 1, 2, 4])
    # Key budget per query block: 512 to 1920 keys, as the listed cases have.
    cap = min(nb + 2, max(3, round(math.exp(rng.uniform(math.log(512), math.log(1920))) / blk)))
    keys = min(L, cap * blk) if kind == "late" else L / 2
    most = {"late": 2.2e9, "dense": 6.5e8, "discover": 2.6e8, "select": 4e9, "diagnose": 2.6e8, "frozen": 3e8}[kind]
    most_rows = 1 << (21 if kind == "late" else 18)  # (batch, head, row) triples
    rows = min(most / keys, most_rows)
    hkv = max(1, min(64 // group, int(rows / (b * L * group) * math.exp(rng.uniform(-2.0, 0.0)))))
    return dict(kind=kind, batch=b, seqlen=L, heads=hkv * group, kv_heads=hkv, dim=d, block=blk, cap=cap,
                sink=rng.choice([0, 1, 1, 2]) if cap > 4 else 1, local=rng.choice([1, 1, 2]) if cap > 4 else 1,
                planted=rng.choice([2, 3, 4, 6]), boost=rng.choice([2.5, 3.0]), std=rng.choice([0.5, 1.0, 1.0]))


def _shape(c):
    return wise.Shape(c["batch"], c["seqlen"], c["heads"], c["kv_heads"], c["dim"], c["block"])


def _select_rule(c):
    return wise.Select(c["sink"], c["local"], wise.WISE_SEL_COVERAGE if c["cap"] % 2 == 0 else wise.WISE_SEL_TOPK,
                       max(0, c["cap"] - c["sink"] - c["local"]), 0.95, c["cap"])


def _planted(c, g):
    """bool [batch, kv heads, nQB, nKB]: key blocks planted in each query block (earlier ones, not the sink)."""
    nb = c["seqlen"] // c["block"]
    q, k = torch.arange(nb, device=DEV)[:, None], torch.arange(nb, device=DEV)[None, :]
    r = torch.rand((c["batch"], c["kv_heads"], nb, nb), generator=g, device=DEV)
    r = r.masked_fill((k < 1) | (k >= q), -1.0)
    top = r.topk(min(c["planted"], nb), dim=-1)
    return torch.zeros_like(r, dtype=torch.bool).scatter_(-1, top.indices, top.values >= 0)


def _support(c, g, planted):
    """Ascending lists padded with -1: sink, local window, planted blocks, others at random up to the cap."""
    nb, cap = c["seqlen"] // c["block"], c["cap"]
    q, k = torch.arange(nb, device=DEV)[:, None], torch.arange(nb, device=DEV)[None, :]
    rank = torch.rand(planted.shape, generator=g, device=DEV) + 2.0 * planted
    rank = rank + 4.0 * ((k < c["sink"]) | (k > q - c["local"]))
    rank = rank.masked_fill(k > q, -1.0)
    top = rank.topk(min(cap, nb), dim=-1)
    blocks = torch.where(top.values >= 0, top.indices, nb).sort(dim=-1).values
    counts = (blocks < nb).sum(-1).to(torch.int32)
    idx = torch.full(planted.shape[:3] + (cap,), -1, dtype=torch.int32, device=DEV)
    idx[..., :blocks.shape[-1]] = torch.where(blocks < nb, blocks, -1).to(torch.int32)
    return idx.contiguous(), counts.contiguous()


def _qkv(c, g, planted, steps):
    """bf16 (Q, K, V) of the given number of recurrent steps."""
    b, L, h, hkv, d, blk = (c[x] for x in ("batch", "seqlen", "heads", "kv_heads", "dim", "block"))
    nb = L // blk
    amp = math.sqrt(c["boost"] * math.sqrt(d))
    sig = torch.randn((b, hkv, nb, d), generator=g, device=DEV)
    sig = amp * sig / sig.norm(dim=-1, keepdim=True)
    x = [torch.randn((b, n, L, d), generator=g, device=DEV) * c["std"] for n in (h, hkv, hkv)]
    x[1].view(b, hkv, nb, blk, d).add_(sig[:, :, :, None])
    x[0].view(b, hkv, h // hkv, nb, blk, d).add_((planted.float() @ sig)[:, :, None, :, None])
    out = []
    for t in range(steps):
        if t:
            for v in x:
                v.add_(torch.randn(v.shape, generator=g, device=DEV), alpha=0.3 * 0.85 ** t)
        out.append(tuple(v.to(torch.bfloat16) for v in x))
    return out


def _masses(c, g, planted, steps):
    """fp32 [steps, batch, heads, nQB, nKB] block masses: each admissible row sums to one, planted blocks and the
    nearest ones hold most."""
    b, h, hkv = c["batch"], c["heads"], c["kv_heads"]
    nb = planted.shape[-1]
    q, k = torch.arange(nb, device=DEV)[:, None], torch.arange(nb, device=DEV)[None, :]
    base = torch.randn((b, h, nb, nb), generator=g, device=DEV)
    base = base + 2.0 * planted.repeat_interleave(h // hkv, 1) + 1.0 * (k == q) + 1.0 * (k == 0)
    base = base.masked_fill(k > q, -math.inf)
    noise = lambda: 0.3 * torch.randn(base.shape, generator=g, device=DEV)  # noqa: E731
    return torch.stack([torch.softmax(base + noise(), -1) for _ in range(steps)]).contiguous()


def _stored_probs(c, q, k, idx, counts):
    """The frozen step's distribution over the support, as wise_freeze_a_probs lays it out (block 128)."""
    b, L, h, hkv, d = (c[x] for x in ("batch", "seqlen", "heads", "kv_heads", "dim"))
    nb, cap = L // 128, idx.shape[-1]
    P = torch.zeros((b, h, nb, cap, 128, 128), dtype=torch.bfloat16, device=DEV)
    inv_l = torch.empty((b, h, nb, 128), device=DEV)
    kb = k.view(b * hkv, nb, 128, d).float()
    qb = q.view(b * hkv, h // hkv, nb, 128, d).float()
    row = torch.arange(128, device=DEV)
    bh = torch.arange(b * hkv, device=DEV)[:, None]
    for i in range(nb):
        li = idx[:, :, i].reshape(b * hkv, cap).long()
        s = torch.einsum("zgrd,zckd->zgrck", qb[:, :, i], kb[bh, li.clamp(min=0)]) / math.sqrt(d)
        keep = (li >= 0)[:, None, :, None] & ((li[:, None, :, None] * 128 + row) <= i * 128 + row[None, :, None, None])
        s = s.masked_fill(~keep[:, None], -math.inf)
        p = torch.exp(s - s.amax((-2, -1), keepdim=True)).to(torch.bfloat16)
        P.view(b * hkv, h // hkv, nb, cap, 128, 128)[:, :, i] = p.transpose(2, 3)
        inv_l.view(b * hkv, h // hkv, nb, 128)[:, :, i] = 1.0 / p.float().sum((-2, -1))
    return P.view(b * h * nb, cap, 128, 128), inv_l.view(b * h * nb, 128)


def prepare(case, seed):
    c, kind, s = case, case["kind"], _shape(case)
    g = torch.Generator(device=DEV).manual_seed(seed)
    nb = s.n_blocks
    planted = _planted(c, g)
    st = {"kind": kind, "shape": s}
    if kind in ("select", "diagnose"):
        masses = _masses(c, g, planted, 4)
        width = nb if kind == "diagnose" else c["cap"]
        st["idx"] = torch.empty((s.batch, s.n_kv_heads, nb, width), dtype=torch.int32, device=DEV)
        st["counts"] = torch.empty((s.batch, s.n_kv_heads, nb), dtype=torch.int32, device=DEV)
        if kind == "select":
            st["mass"], st["rule"] = masses.sum(0), _select_rule(c)
        else:
            st["masses"], st["running"] = masses, _support(c, g, planted)
            st["retained"] = torch.empty((s.batch, s.n_heads, nb), device=DEV)
            st["overlap"] = torch.empty((s.batch, 2), dtype=torch.int64, device=DEV)
        return st
    st["qkv"] = _qkv(c, g, planted, 2 if kind == "discover" else 1)
    st["O"] = [torch.empty_like(q) for q, _, _ in st["qkv"]]
    if kind in ("late", "frozen"):
        st["idx"], st["counts"] = _support(c, g, planted)
    if kind == "discover":
        st["mass"] = torch.empty((s.batch, s.n_heads, nb, nb), device=DEV)
    if kind == "frozen":
        q, k, _ = st["qkv"][0]
        cap = wise.freeze_tile_cap(s, c["cap"])
        width = max(1, int(st["counts"].max()))
        P, st["inv_l"] = _stored_probs(c, q, k, st["idx"][..., :width], st["counts"])
        st["P"] = torch.zeros((P.shape[0], cap, 128, 128), dtype=torch.bfloat16, device=DEV)
        st["P"][:, :width] = P
    return st


def run(state):
    kind, s = state["kind"], state["shape"]
    if kind == "late":
        (q, k, v), o = state["qkv"][0], state["O"][0]
        wise.wise_sparse_attn(s, q, k, v, state["idx"], state["counts"], o)
        return o
    if kind == "dense":
        (q, k, v), o = state["qkv"][0], state["O"][0]
        wise.wise_full_attn_accumulate(s, q, k, v, o)
        return o
    if kind == "discover":
        for t, ((q, k, v), o) in enumerate(zip(state["qkv"], state["O"])):
            wise.wise_full_attn_accumulate(s, q, k, v, o, state["mass"], t)
        return {"O": state["O"], "mass": state["mass"]}
    if kind == "select":
        wise.wise_select_support(s, state["rule"], state["mass"], state["idx"], state["counts"])
        return {"idx": state["idx"], "counts": state["counts"]}
    if kind == "diagnose":
        ri, rc = state["running"]
        wise.wise_select_working_set(s, wise.WS_UNION, state["masses"], state["idx"], state["counts"])
        wise.wise_support_mass(s, state["masses"][-1], ri, rc, state["retained"])
        wise.wise_support_overlap(s, state["idx"], state["counts"], ri, rc, state["overlap"])
        return {"idx": state["idx"], "counts": state["counts"], "retained": state["retained"],
                "overlap": state["overlap"]}
    (_, _, v), o = state["qkv"][0], state["O"][0]
    wise.wise_frozen_pv(s, state["P"], state["inv_l"], v, state["idx"], state["counts"], o)
    return o


def _pairs(c, kind):
    """(query, key) pairs of one head that the path computes."""
    L, blk = c["seqlen"], c["block"]
    if kind in ("late", "frozen"):
        nb = L // blk
        return sum((min(q + 1, c["cap"]) - 1) * blk * blk + blk * (blk + 1) // 2 for q in range(nb))
    return L * (L + 1) // 2


def work(case):
    c, kind = case, case["kind"]
    b, L, h, hkv, d = (c[x] for x in ("batch", "seqlen", "heads", "kv_heads", "dim"))
    nb = L // c["block"]
    tri, lists = nb * (nb + 1) // 2, b * hkv * nb
    if kind == "select":
        return {"bytes": 4 * b * h * tri + 4 * lists * (c["cap"] + 1), "flops": b * h * tri}
    if kind == "diagnose":
        kept = sum(min(q + 1, c["cap"]) for q in range(nb))
        return {"bytes": 4 * 4 * b * h * tri + 4 * lists * (nb + 1) + 4 * b * hkv * kept + 4 * b * h * nb,
                "flops": 4 * b * h * tri + b * h * kept}
    qo, kv = 2 * b * h * L * d, 2 * b * hkv * L * d
    pairs = b * h * _pairs(c, kind)
    if kind == "frozen":
        tiles = b * h * sum(min(q + 1, c["cap"]) for q in range(nb))
        return {"bytes": tiles * 32768 + 4 * b * h * L + kv + qo + 4 * lists * c["cap"], "flops": 2 * d * pairs}
    steps = 2 if kind == "discover" else 1
    bytes_ = steps * (2 * qo + 2 * kv)
    if kind == "late":
        bytes_ += 4 * lists * (c["cap"] + 1)
    if kind == "discover":
        bytes_ += 4 * b * h * nb * nb
    return {"bytes": bytes_, "flops": steps * 4 * d * pairs}


def _exact_full(c, q, k, v, mass):
    """Causal attention of one step in 64 bits, and its block mass if asked for."""
    b, L, h, hkv, d, blk = (c[x] for x in ("batch", "seqlen", "heads", "kv_heads", "dim", "block"))
    nb = L // blk
    o = torch.empty((b, h, L, d), dtype=torch.float64, device=DEV)
    r = torch.empty((b, h, nb, nb), dtype=torch.float64, device=DEV) if mass else None
    future = torch.ones((L, L), dtype=torch.bool, device=DEV).triu(1)
    for i in range(b):
        for j in range(h):
            g = j // (h // hkv)
            a = (q[i, j].double() @ k[i, g].double().T / math.sqrt(d)).masked_fill_(future, -math.inf).softmax(-1)
            o[i, j] = a @ v[i, g].double()
            if mass:
                r[i, j] = a.view(nb, blk, nb, blk).sum((1, 3)) / blk
    return o, r


def _exact_late(c, q, k, v, idx):
    """Support-restricted attention in 64 bits, one query block of every head at a time."""
    b, L, h, hkv, d, blk = (c[x] for x in ("batch", "seqlen", "heads", "kv_heads", "dim", "block"))
    nb, cap, z = L // blk, idx.shape[-1], b * hkv
    qb, kb, vb = q.view(z, h // hkv, nb, blk, d), k.view(z, nb, blk, d), v.view(z, nb, blk, d)
    o = torch.empty((z, h // hkv, nb, blk, d), dtype=torch.float64, device=DEV)
    row = torch.arange(blk, device=DEV)
    for i in range(nb):
        for z0 in range(0, z, 32):
            zs = slice(z0, min(z, z0 + 32))
            li = idx.view(z, nb, cap)[zs, i].long()
            at = torch.arange(zs.start, zs.stop, device=DEV)[:, None]
            ks, vs = (x[at, li.clamp(min=0)].flatten(1, 2).double() for x in (kb, vb))
            key = (li[:, :, None] * blk + row).flatten(1)
            keep = (key >= 0)[:, None] & (key[:, None] <= i * blk + row[:, None])
            keep &= (li >= 0).repeat_interleave(blk, 1)[:, None]
            s = (qb[zs, :, i].double() @ ks[:, None].transpose(-1, -2) / math.sqrt(d))
            o[zs, :, i] = s.masked_fill_(~keep[:, None], -math.inf).softmax(-1) @ vs[:, None]
    return o.view(b, h, L, d)


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "select":
        return None  # whole numbers only
    g = torch.Generator(device=DEV).manual_seed(seed)
    planted = _planted(c, g)
    b, L, h, hkv = c["batch"], c["seqlen"], c["heads"], c["kv_heads"]
    if kind == "diagnose":
        last = _masses(c, g, planted, 4)[-1].double()
        idx, _ = _support(c, g, planted)
        li = idx.repeat_interleave(h // hkv, 1).long()
        kept = last.gather(-1, li.clamp(min=0)).masked_fill(li < 0, 0.0).sum(-1)
        return {"idx": None, "counts": None, "retained": kept, "overlap": None}
    qkv = _qkv(c, g, planted, 2 if kind == "discover" else 1)
    if kind == "dense":
        return _exact_full(c, *qkv[0], False)[0]
    if kind == "discover":
        outs = [_exact_full(c, *x, True) for x in qkv]
        return {"O": [o for o, _ in outs], "mass": outs[0][1] + outs[1][1]}
    idx, counts = _support(c, g, planted)
    if kind == "late":
        return _exact_late(c, *qkv[0], idx)
    q, k, v = qkv[0]
    nb, cap = L // 128, max(1, int(counts.max()))
    P, inv_l = _stored_probs(c, q, k, idx[..., :cap], counts)
    P, d = P.view(b * hkv, h // hkv, nb, cap, 128, 128), c["dim"]
    o = torch.empty((b * hkv, h // hkv, nb, 128, d), dtype=torch.float64, device=DEV)
    vb = v.view(b * hkv, nb, 128, d)
    at = torch.arange(b * hkv, device=DEV)[:, None]
    for i in range(nb):
        li = idx.view(b * hkv, nb, -1)[:, i, :cap].long()
        o[:, :, i] = torch.einsum("zgcrk,zckd->zgrd", P[:, :, i].double(), vb[at, li.clamp(min=0)].double())
    o *= inv_l.view(b * hkv, h // hkv, nb, 128, 1).double()
    return o.view(b, h, L, d)
