"""The work that programs have this library do, as measurable cases.

One pass is one decode step of one attention layer, or of one layer of each
of several co-located models: the new tokens' K/V rows are appended to the
paged pool and every sequence's query attends over its context, through the
entry point that such a program calls.  A case's lengths are the quantiles of
its distribution, so that its work depends on the case alone; the seed sets
which sequence has which length, where the blocks lie, and all values.  A pass
does not advance the lengths, so it can be repeated: it appends the same rows
to the same slots again.
"""
from __future__ import annotations

import math
from statistics import NormalDist

import numpy as np
import torch

from paper_2606_12950_gb300 import kvpool as K
from paper_2606_12950_gb300.runner import DevicePool

# how a program makes the step:
#   append+attend    kv_append, then paged_decode_attn
#   append_attend    paged_decode_attn_append (fused)
#   attend           paged_decode_attn, the rows being in the pool already
#   noalloc          the same without a workspace of the caller's
#   seqtab           paged_decode_attn_seqtab: the host sequence table's sync,
#                    the append and the attention in one call
#   cascade          paged_decode_attn_cascade: groups of sequences, each
#                    sharing a prefix by reference, fused append
#   cascade_seqtab   the same with the host sequence table's sync
#   multi            paged_decode_attn_multi: co-located models in one pool
APPENDS = ("append+attend", "append_attend", "seqtab", "cascade", "cascade_seqtab", "multi")


def _case(name, call, seqs, heads, lens, *, head_dim=128, block=16, mid=0, alpha=0.0, lo=1, hi=0, groups=0, prefix=0,
          overlap=False, host_io=False):
    """heads: query x KV heads of a layer; for several co-located models one
    such pair each, with `seqs` their numbers of sequences."""
    c = {"call": call, "seqs": str(seqs), "heads": heads, "head_dim": head_dim, "block": block, "lens": lens,
         "mid": mid, "alpha": alpha, "lo": lo, "hi": hi, "groups": groups, "prefix": prefix, "overlap": overlap,
         "host_io": host_io}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest model of the tests, 4 short contexts, append and
        # attention as two calls: launches and latency
        _case("tiny_two_calls", "append+attend", 4, "4x2", "18,65,101,256", head_dim=64),
        # one user's chat with a long history: a single sequence on the whole GPU
        _case("one_long_chat", "append_attend", 1, "32x8", "equal", mid=8193),
        # a lightly loaded server: a few agents of a 40-head model, ragged contexts
        _case("eight_agents", "append_attend", 8, "40x8", "uniform", lo=601, hi=3500),
        # the benchmark's ordinary batch, driven by the host sequence table,
        # steps back to back with the step overlap that a decode loop turns on
        _case("ordinary_batch", "seqtab", 64, "32x8", "lognormal", mid=1024, hi=16384, overlap=True),
        # the same batch with inputs and outputs in pinned host memory
        _case("ordinary_batch_host_io", "seqtab", 64, "32x8", "lognormal", mid=1024, hi=16384, overlap=True,
              host_io=True),
        # a small model's 64-wide heads, many sequences, blocks of 32 tokens
        _case("head64_batch", "append_attend", 128, "32x8", "lognormal", head_dim=64, block=32, mid=1000, hi=16384),
        # a model without grouped heads: 32 KV heads, no sharing of K/V reads
        _case("mha_batch", "append_attend", 30, "32x32", "uniform", lo=333, hi=2100),
        # eight query heads per KV head, by a server that gave all its memory
        # to the pool and has no workspace to hand over
        _case("wide_group_noalloc", "noalloc", 48, "64x8", "lognormal", block=32, mid=1500, hi=16384),
        # Planner -> Coder -> Reviewer chains over one shared system prompt
        _case("agent_chains", "cascade_seqtab", 256, "32x8", "lognormal", mid=300, hi=8192, groups=1, prefix=2048,
              overlap=True),
        # three roles with long instructions of their own, and short outputs so far
        _case("role_prompts", "cascade", 190, "32x8", "lognormal", mid=300, hi=4096, groups=3, prefix=4096),
        # three co-located models decoding from one pool
        _case("colocated_models", "multi", "205,205,102", "32x32,32x8,40x8", "pareto", alpha=1.5, lo=128, hi=32768),
        # long contexts with a heavy tail, the largest batch
        _case("long_context", "seqtab", 1024, "32x8", "pareto", block=32, alpha=1.2, lo=256, hi=131072, overlap=True),
    ]


# K/V bytes of the largest listed case, about: a drawn case stays below
_MOST_BYTES = 4.0e9


def draw(rng):
    """A case of the same ranges: 1 to 1024 sequences of 16 to 65536 tokens,
    head dims, groups, blocks and calls as listed."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    call = rng.choice(["append+attend", "append_attend", "append_attend", "attend", "noalloc", "seqtab", "seqtab",
                       "cascade", "cascade_seqtab", "multi"])
    head_dim = rng.choice([64, 128, 128, 128])
    block = rng.choice([16, 16, 32, 64])
    overlap = call in ("seqtab", "cascade", "cascade_seqtab") and rng.random() < 0.5
    lens, alpha = rng.choice(["equal", "uniform", "lognormal", "pareto"]), rng.choice([1.2, 1.5])
    if call == "multi":
        n = log_int(3, 300)
        shapes = rng.sample(["32x32", "32x8", "40x8", "16x2", "64x8"], rng.choice([2, 3]))
        seqs = ",".join(str(max(1, int(n * rng.uniform(0.3, 1.0)))) for _ in shapes)
        return _shrunk(_case("", call, seqs, ",".join(shapes), lens, block=16, mid=log_int(64, 4096), alpha=alpha,
                             lo=rng.randrange(16, 400), hi=log_int(512, 32768)))
    seqs = log_int(1, 1024)
    kv = rng.choice([1, 2, 4, 8, 8, 8, 32])
    group = 1 if kv == 32 else rng.choice([1, 2, 4, 4, 5, 8])
    heads = "%dx%d" % (kv * group, kv)
    if call.startswith("cascade"):
        seqs = max(2, seqs)
        groups = rng.randrange(1, min(6, seqs) + 1)
        prefix = 64 * log_int(2, 128)
        return _shrunk(_case("", call, seqs, heads, lens, head_dim=head_dim, block=block, mid=log_int(16, 2048),
                             alpha=alpha, lo=rng.randrange(1, 300), hi=log_int(512, 8192), groups=groups, prefix=prefix,
                             overlap=overlap))
    c = _shrunk(_case("", call, seqs, heads, lens, head_dim=head_dim, block=block, mid=log_int(16, 16384), alpha=alpha,
                      lo=rng.randrange(16, 700), hi=log_int(1024, 65536), overlap=overlap,
                      host_io=call == "seqtab" and rng.random() < 0.25))
    if call == "noalloc":  # the library's own scratch is 32 MiB
        record = (group * head_dim + 2 * group + 3) // 4 * 16
        if (int(c["seqs"]) * kv + 4096) * record > 24 << 20:
            c["call"] = "attend"
    return c


def _shrunk(c):
    """Fewer sequences until the case reads no more than the largest listed one."""
    while work(c)["bytes"] > _MOST_BYTES:
        c["seqs"] = ",".join(str(max(c["groups"], 1, int(n) * 3 // 4)) for n in c["seqs"].split(","))
        if all(int(n) <= max(c["groups"], 1) for n in c["seqs"].split(",")):
            c["hi"], c["mid"] = max(64, c["hi"] // 2), max(64, c["mid"] // 2)
    return c


def _lengths(case, n):
    """The quantiles of the case's lengths, smallest first; with a shared
    prefix the lengths after it."""
    kind, lo, hi, mid = case["lens"], case["lo"], case["hi"], case["mid"]
    if "," in kind:
        return np.array([int(x) for x in kind.split(",")], dtype=np.int64)
    hi = max(hi, lo)
    u = (np.arange(n) + 0.5) / n
    if kind == "equal":
        x = np.full(n, float(mid))
    elif kind == "uniform":
        x = lo + u * (hi - lo)
    elif kind == "lognormal":  # sigma = 1
        x = np.clip(mid * np.exp([NormalDist().inv_cdf(v) for v in u]), lo, hi)
    else:  # bounded Pareto
        a = case["alpha"]
        x = lo / np.power(1.0 - u * (1.0 - (lo / hi) ** a), 1.0 / a)
    return np.maximum(1, np.floor(x)).astype(np.int64)


def _batches(case):
    """(sequences, query heads, KV heads) of each model's batch."""
    return [(int(n),) + tuple(int(h) for h in heads.split("x"))
            for n, heads in zip(case["seqs"].split(","), case["heads"].split(","))]


def work(case):
    d, bs, nbytes, flops = case["head_dim"], case["block"], 0, 0
    for S, Hq, Hkv in _batches(case):
        lens = _lengths(case, S)
        row = 2 * Hkv * d * 2  # K and V of one token
        read = int(lens.sum()) + case["groups"] * case["prefix"]  # a shared prefix is read once
        nbytes += read * row + 2 * S * Hq * d * 2 + 4 * S + 4 * int((-(-lens // bs)).sum())
        if case["call"] == "append+attend":
            nbytes += 2 * S * row
        elif case["call"] in APPENDS:
            nbytes += S * row  # the new token's rows are read from the input and written
        flops += 4 * Hq * d * (int(lens.sum()) + S * (case["prefix"] if case["groups"] else 0))
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # bf16 outputs of fp32 sums, the softmax weights rounded to bf16 for the
    # tensor cores: about 2.5e-3 from the 64-bit result (2-norm)
    return {"rel": 1e-2, "max": 6e-2}


class _State:
    pass


def _rows(shape, g, host_io):
    t = torch.randn(shape, generator=g, device="cuda").to(torch.bfloat16)
    if not host_io:
        return t
    h = torch.empty(shape, dtype=torch.bfloat16, pin_memory=True)
    h.copy_(t)
    return h


def prepare(case, seed):
    st = _State()
    st.case = case
    d, bs, groups, prefix = case["head_dim"], case["block"], case["groups"], case["prefix"]
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    rng = np.random.default_rng(seed)
    shapes = _batches(case)
    lens = [rng.permutation(_lengths(case, S)) for S, _, _ in shapes]
    shared = prefix if groups else 0  # tokens, whole blocks
    page_bytes = min(2 * Hkv * bs * d * 2 for _, _, Hkv in shapes)
    n_pages = 0
    for (S, _, Hkv), n in zip(shapes, lens):
        blocks = int((-(-n // bs)).sum()) + groups * shared // bs
        n_pages += (blocks + blocks // 9 + 8) * (2 * Hkv * bs * d * 2 // page_bytes)  # about 90% full
    n_pages = -(-n_pages // 64) * 64
    st.pool = DevicePool(n_pages, page_bytes, bs, [(Hkv, d) for _, _, Hkv in shapes], shuffle_seed=seed + 1)
    st.pool.buf.view(torch.bfloat16).normal_(generator=g)
    if case["overlap"]:
        st.pool.set_step_overlap(True)
    st.batches = []
    for layout, ((S, Hq, Hkv), n) in enumerate(zip(shapes, lens)):
        b = _State()
        b.layout, b.S, b.Hq, b.Hkv, b.scale = layout, S, Hq, Hkv, d ** -0.5
        total = n + shared
        b.max_blocks = int(-(-total.max() // bs))
        rows = S
        member_of = np.arange(S) * groups // S if groups else None
        if case["call"] in ("seqtab", "cascade_seqtab"):
            # each group's prefix is held by a slot of its own after the decode rows
            rows = S + groups
            b.tab = K.SeqTab(st.pool.handle, layout, rows, b.max_blocks)
            for k in range(groups):
                b.tab.reserve(S + k, prefix)
                b.tab.set_len(S + k, prefix)
            for s in range(S):
                if groups:
                    b.tab.share_prefix(s, S + int(member_of[s]), prefix // bs)
                b.tab.reserve(s, int(total[s]))
                b.tab.set_len(s, int(total[s]))
        else:
            table = np.full((S, b.max_blocks), -1, dtype=np.int32)
            heads = [K.kv_alloc_blocks(st.pool.handle, layout, prefix // bs) for _ in range(groups)]
            for s in range(S):
                if groups:
                    table[s, : shared // bs] = heads[int(member_of[s])]
                nb = int(-(-total[s] // bs))
                table[s, shared // bs : nb] = K.kv_alloc_blocks(st.pool.handle, layout, nb - shared // bs)
        b.table = torch.empty((rows, b.max_blocks), dtype=torch.int32, device="cuda")
        b.lens = torch.empty(rows, dtype=torch.int32, device="cuda")
        if case["call"] in ("seqtab", "cascade_seqtab"):
            b.tab.sync(b.table, b.lens)
        else:
            K.kv_block_table_upload(st.pool.handle, layout, table, total, b.table, b.lens)
        b.q = _rows((S, Hq, d), g, case["host_io"])
        b.k_new = _rows((S, Hkv, d), g, case["host_io"])
        b.v_new = _rows((S, Hkv, d), g, case["host_io"])
        b.out = torch.zeros((S, Hq, d), dtype=torch.bfloat16, device="cpu" if case["host_io"] else "cuda",
                            pin_memory=case["host_io"])
        b.ws, b.ws_bytes = None, 0
        if case["call"] != "noalloc":
            size = K.kv_cascade_workspace_bytes if groups else K.kv_workspace_bytes
            b.ws_bytes = max(256, size(st.pool.handle, layout, S, Hq, b.max_blocks))
            b.ws = torch.empty(b.ws_bytes, dtype=torch.uint8, device="cuda")
        if groups:
            b.plan = K.PrefixPlan([(np.nonzero(member_of == k)[0].tolist(), prefix) for k in range(groups)])
        st.batches.append(b)
    if case["call"] == "multi":
        st.multi = K.attn_batches([{
            "layout": b.layout, "q": b.q, "k_new": b.k_new, "v_new": b.v_new, "out": b.out, "dev_table": b.table,
            "dev_ctx_lens": b.lens, "max_blocks": b.max_blocks, "S": b.S, "Hq": b.Hq, "scale": b.scale,
            "workspace": b.ws, "ws_bytes": b.ws_bytes} for b in st.batches])
    return st


def run(st):
    call, h, b = st.case["call"], st.pool.handle, st.batches[0]
    if call == "append+attend":
        K.kv_append(h, 0, b.k_new, b.v_new, b.table, b.lens, b.max_blocks, b.S)
        K.paged_decode_attn(h, 0, b.q, b.out, b.table, b.lens, b.max_blocks, b.S, b.Hq, b.scale, 0, b.ws, b.ws_bytes)
    elif call == "append_attend":
        K.paged_decode_attn_append(h, 0, b.q, b.k_new, b.v_new, b.out, b.table, b.lens, b.max_blocks, b.S, b.Hq,
                                   b.scale, 0, b.ws, b.ws_bytes)
    elif call == "attend":
        K.paged_decode_attn(h, 0, b.q, b.out, b.table, b.lens, b.max_blocks, b.S, b.Hq, b.scale, 0, b.ws, b.ws_bytes)
    elif call == "noalloc":
        K.paged_decode_attn_noalloc(h, 0, b.q, b.out, b.table, b.lens, b.max_blocks, b.S, b.Hq, b.scale)
    elif call == "seqtab":
        K.paged_decode_attn_seqtab(h, b.tab, b.q, b.k_new, b.v_new, b.out, b.table, b.lens, b.S, b.Hq, b.scale, 0,
                                   b.ws, b.ws_bytes)
    elif call == "cascade":
        K.paged_decode_attn_cascade(h, 0, b.q, b.k_new, b.v_new, b.out, b.table, b.lens, b.max_blocks, b.S, b.Hq,
                                    b.scale, b.plan, b.ws, b.ws_bytes)
    elif call == "cascade_seqtab":
        K.paged_decode_attn_cascade_seqtab(h, b.tab, b.q, b.k_new, b.v_new, b.out, b.table, b.lens, b.S, b.Hq,
                                           b.scale, b.plan, b.ws, b.ws_bytes)
    else:
        K.paged_decode_attn_multi(h, st.multi)
    out = {"out%d" % i: b.out for i, b in enumerate(st.batches)}
    if call in APPENDS:  # the pool that the step appended to
        out["pool"] = st.pool.buf.view(torch.bfloat16)
    if call in ("seqtab", "cascade_seqtab"):
        out["lens"], out["table"] = b.lens, b.table
    return out


def exact(case, seed):
    st = prepare(case, seed)
    torch.cuda.synchronize()
    d, bs = case["head_dim"], case["block"]
    call, pool, page = case["call"], st.pool.buf.view(torch.bfloat16), st.pool.page_bytes // 2
    out = {}
    for i, b in enumerate(st.batches):
        elems = 2 * b.Hkv * bs * d  # of a block, which starts at its first page
        lens, S = b.lens[: b.S].long(), b.S
        q, kn, vn = (t.cuda() for t in (b.q, b.k_new, b.v_new))
        inside = torch.arange(elems, device="cuda").view(2, b.Hkv, bs, d)
        if call in APPENDS:
            pos = lens - 1
            blk = b.table[torch.arange(S, device="cuda"), pos // bs].long()
            for kv, new in ((0, kn), (1, vn)):
                at = blk.view(S, 1, 1) * page + inside[kv].permute(1, 0, 2)[pos % bs]
                pool[at.reshape(-1)] = new.reshape(-1)
        o = torch.empty((S, b.Hq, d), dtype=torch.float64, device="cuda")
        for s, n in enumerate(lens.tolist()):
            ids = b.table[s, : -(-n // bs)].long()
            if elems % page == 0 and elems > page:
                at = ids.view(-1, 1) + torch.arange(elems // page, device="cuda")
            else:
                at = ids.view(-1, 1)
            kv = pool.view(-1, page)[at.reshape(-1)].view(-1, 2, b.Hkv, bs, d).permute(1, 2, 0, 3, 4)
            kv = kv.reshape(2, b.Hkv, -1, d)[:, :, :n].double()
            w = torch.softmax(q[s].double().view(b.Hkv, -1, d) @ kv[0].transpose(1, 2) * b.scale, dim=-1)
            o[s] = (w @ kv[1]).view(b.Hq, d)
        out["out%d" % i] = o
    if call in APPENDS:
        out["pool"] = pool.double()
    if call in ("seqtab", "cascade_seqtab"):
        out["lens"], out["table"] = None, None
    return out
