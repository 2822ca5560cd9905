"""Decode-attention cases over the range the library is used for, each one pass through its public calls.

A case is one call (or the pair of calls) a generation loop makes per decode step and layer: references or span lists
in, attention rows out, or the full-context attention of a "determine span" step.  Sizes are those of the
repository's workloads (batch 1 to 64, 8 or 32 heads of 64 or 128, contexts of 256 to 16384 tokens, 1 to 50 per cent
of them selected) and of its variants: grouped query heads, several query tokens, an 8-bit and a paged cache, the
blocked encoding, a step driven from host buffers.  Queries, keys and values are N(0, 1), as in the repository's tests.

`how` names the calls:
  step       ssa_decode_step, everything resident: span lists -> index lists and attention
  host_step  ssa_decode_step with the step's inputs and results in pinned host memory
  refs       ssa_refs_to_index, then ssa_decode_attn_sparse
  sparse     ssa_decode_attn_sparse on index lists in hand (every layer of a model after the first)
  paged      ssa_decode_attn_sparse_paged on index lists in hand
  blockmask  ssa_spans_to_blockmask, then ssa_decode_attn_blockmask
  dense      ssa_decode_attn_dense, the full context
  multiq     ssa_decode_attn_dense_multiq, several query tokens over the full context
"""
import math

import numpy as np
import torch

from paper_2404_09336_b200 import ssa

DTYPES = {"bf16": torch.bfloat16, "f16": torch.float16, "fp8": torch.float8_e4m3fn}
MAX_CACHE_BYTES = 4 << 30          # K and V of the largest listed case ...
MAX_FLOPS = 4.5e9                  # ... and about its operations
LINE = 40                          # tokens of one referenced line


def _case(name, how, B, H, D, ctx, dtype, **more):
    """ctx_lo: context lengths are uniform in [ctx_lo, ctx].  Spans: [0, prefix), the last `tail` tokens, and either
    spans_lo..spans_hi spans (lines for `refs`) of len_lo..len_hi tokens, or spans of 16..256 tokens until a
    fraction `density` of the context is selected.  full_every = k: every k-th request attends to its full context."""
    c = {"how": how, "B": B, "H": H, "H_kv": H, "D": D, "ctx": ctx, "ctx_lo": ctx, "dtype": dtype, "prefix": 64,
         "tail": 64, "spans_lo": 0, "spans_hi": 0, "len_lo": 0, "len_hi": 0, "density": 0.0, "full_every": 0, "n_q": 1,
         "page_size": 0, "block_size": 0}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    arithmetic = dict(ctx_lo=256, tail=32, spans_lo=1, spans_hi=4, len_lo=4, len_hi=32)
    return [
        # one short request, few small heads, half precision: the least work a decode step can have, all latency
        _case("tiny_step", "step", 1, 8, 64, 512, "f16", prefix=32, tail=16, spans_lo=3, spans_hi=3, len_lo=8, len_hi=16),
        # arithmetic traces: a large batch of short ragged contexts, a few short spans each
        _case("arithmetic_step", "step", 64, 32, 128, 1024, "bf16", **arithmetic),
        # the same step driven from pinned host buffers: new queries and spans in, rows out, every step
        _case("arithmetic_host_step", "host_step", 64, 32, 128, 1024, "bf16", **arithmetic),
        # summarization: the model's references to article lines resolved on the device, then attention
        _case("summarization_refs", "refs", 16, 32, 128, 4096, "bf16", spans_lo=2, spans_hi=10, len_lo=1, len_hi=5),
        # few requests with long contexts and long spans
        _case("long_context_step", "step", 8, 32, 128, 16384, "bf16", tail=128, spans_lo=16, spans_hi=16, len_lo=32, len_hi=256),
        # a batch in which every eighth request is at a "determine span" step and attends to all of its context
        _case("mixed_step", "step", 64, 32, 128, 1024, "bf16", full_every=8, **arithmetic),
        # the paper's kernel micro-benchmark: half of the tokens ignored, in its blocked (index, bitmask) encoding
        _case("microbench_blockmask", "blockmask", 64, 32, 128, 2048, "bf16", prefix=0, density=0.5, block_size=256),
        # a later layer of a model with grouped query heads: the index lists exist already
        _case("grouped_heads_layer", "sparse", 32, 32, 128, 8192, "bf16", H_kv=8, prefix=0, density=0.10),
        # four query tokens per request (speculative decoding) over ragged full contexts, grouped query heads
        _case("grouped_multi_token_dense", "multiq", 17, 32, 128, 8190, "bf16", H_kv=8, ctx_lo=1001, n_q=4),
        # an 8-bit cache, as kept for long contexts by models with grouped query heads
        _case("fp8_grouped_step", "step", 32, 32, 128, 8192, "fp8", H_kv=8, prefix=0, density=0.10),
        # a serving stack's paged cache, index lists in hand
        _case("paged_layer", "paged", 64, 32, 128, 1024, "bf16", page_size=16, **arithmetic),
        # "determine span" step of a large batch: every request reads its whole context; the largest call
        _case("determine_span_dense", "dense", 32, 32, 128, 8192, "bf16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    how = rng.choice(["step", "step", "step", "host_step", "refs", "sparse", "sparse", "blockmask", "dense", "multiq", "paged"])
    D = rng.choice([64, 128, 128, 128])
    dtype = rng.choice(["bf16", "bf16", "f16"])
    H = rng.choice([8, 32, 32])
    B = _log_int(rng, 1, 64)
    ctx = _log_int(rng, 256, 16384)
    more = dict(ctx_lo=rng.choice([ctx, max(1, ctx // 4)]))
    if how in ("step", "sparse", "dense", "multiq") and rng.random() < (1.0 if how == "multiq" else 0.5):
        H, D = 32, 128
        more["H_kv"] = rng.choice([4, 8, 8])
    if how in ("step", "sparse") and rng.random() < 0.3:
        dtype = "fp8"
    if how == "multiq":
        more["n_q"] = rng.randint(2, 4)
    if how == "host_step":
        ctx = min(ctx, 2048)
        more["ctx_lo"] = max(1, ctx // 4)
    if how == "refs":
        more.update(spans_lo=2, spans_hi=rng.randint(3, 12), len_lo=1, len_hi=5)
        ctx = max(ctx, 1024)
        more["ctx_lo"] = max(1024, more["ctx_lo"])
    elif how not in ("dense", "multiq"):
        if rng.random() < 0.5 and how != "blockmask":
            longest = max(8, ctx // 32)
            more.update(spans_lo=1, spans_hi=rng.randint(2, 20), len_lo=4, len_hi=longest, tail=32)
        else:
            more.update(prefix=0, density=round(math.exp(rng.uniform(math.log(0.01), math.log(0.5))), 4))
        if how == "step" and rng.random() < 0.2:
            more["full_every"] = rng.choice([2, 4, 8])
    if how == "paged":
        more["page_size"] = rng.choice([16, 32, 64])
    if how == "blockmask":
        more["block_size"] = rng.choice([64, 128, 256])
    c = _case(None, how, B, H, D, ctx, dtype, **more)
    while c["B"] > 1 and (c["B"] * c["ctx"] * _cache_row_bytes(c) > MAX_CACHE_BYTES
                          or c["B"] * c["ctx"] * c["H"] * c["n_q"] * c["D"] * 4.0 > MAX_FLOPS):
        c["B"] //= 2
    return c


def _cache_row_bytes(c):
    """K + V bytes of one cached position over all cache heads."""
    return 2 * c["H_kv"] * c["D"] * DTYPES[c["dtype"]].itemsize


# ---- span lists -------------------------------------------------------------------------------------------------
def _spans_of_request(r, c, b, n):
    if c["full_every"] and b % c["full_every"] == 0:
        return [(0, n)]
    if c["density"]:
        target = max(1, int(round(c["density"] * n)))
        tail = min(c["tail"], target)
        lengths, left = [], target - tail
        while left > 0:
            ln = min(int(r.integers(16, 257)), left)
            lengths.append(ln)
            left -= ln
        # disjoint: the unselected tokens in front of the tail fall into the gaps at random
        cuts = np.sort(r.integers(0, n - target + 1, size=len(lengths)))
        spans, used = [], 0
        for cut, ln in zip(cuts.tolist(), lengths):
            spans.append((cut + used, cut + used + ln))
            used += ln
        spans.append((n - tail, n))
    else:
        spans = [(0, min(c["prefix"], n)), (max(n - c["tail"], 0), n)]
        for _ in range(int(r.integers(c["spans_lo"], c["spans_hi"] + 1))):
            ln = int(r.integers(c["len_lo"], c["len_hi"] + 1))
            s = int(r.integers(0, max(n - ln, 0) + 1))
            spans.append((s, min(s + ln, n)))
    return [spans[i] for i in r.permutation(len(spans))]


def _most_selected(c):
    """The most positions a request of this case can attend to: what its index buffers are allocated for."""
    if c["full_every"]:
        return c["ctx"]
    if c["density"]:
        return max(1, int(round(c["density"] * c["ctx"])))
    span = c["len_hi"] * (LINE if c["how"] == "refs" else 1)
    return min(c["ctx"], c["prefix"] + c["tail"] + LINE + c["spans_hi"] * span)


def _lines_of_request(r, c, n):
    """Completed lines behind the prefix, references to ranges of them, and the start of the current line."""
    first, last = c["prefix"], n - c["tail"]
    lines = [(s, min(s + LINE, last)) for s in range(first, last, LINE)]
    refs = []
    for _ in range(int(r.integers(c["spans_lo"], c["spans_hi"] + 1))):
        count = min(int(r.integers(c["len_lo"], c["len_hi"] + 1)), len(lines))
        lo = int(r.integers(0, len(lines) - count + 1))
        refs.append((lo, lo + count - 1))
    return lines, refs, last


def _lists(c, seed):
    r = np.random.Generator(np.random.PCG64([int(seed), 77]))
    ctx = r.integers(c["ctx_lo"], c["ctx"] + 1, size=c["B"]).astype(np.int32)
    out = {"ctx": ctx}
    if c["how"] in ("dense", "multiq"):
        out["selected"] = ctx.astype(np.int64)
    elif c["how"] == "refs":
        out["lines"], out["refs"], out["line_start"] = zip(*(_lines_of_request(r, c, int(n)) for n in ctx))
        spans = [_request_spans(c, out, b) for b in range(c["B"])]
    else:
        spans = out["spans"] = [_spans_of_request(r, c, b, int(n)) for b, n in enumerate(ctx)]
    if "selected" not in out:
        out["bound"] = max(1, min(c["ctx"], max(sum(e - s for s, e in sp) for sp in spans)))
        out["max_spans"] = max(len(sp) for sp in spans)
        sel = []
        for sp, n in zip(spans, ctx):
            hit = np.zeros(int(n), bool)
            for s, e in sp:
                hit[s:e] = True
            sel.append(int(hit.sum()))
        out["selected"] = np.asarray(sel, np.int64)
    return out


def _offsets(lists):
    return np.concatenate([[0], np.cumsum([len(x) for x in lists])]).astype(np.int32)


def _pairs(lists):
    return np.asarray([p for x in lists for p in x], np.int32).reshape(-1, 2)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# ---- state ------------------------------------------------------------------------------------------------------
def _normal(shape, dtype, gen):
    if dtype != torch.float8_e4m3fn:
        return torch.empty(shape, dtype=dtype, device="cuda").normal_(generator=gen)
    out = torch.empty(shape, dtype=dtype, device="cuda")
    for i in range(shape[0]):      # no 8-bit generator: one request at a time through 16 bits
        out[i] = torch.empty(shape[1:], dtype=torch.bfloat16, device="cuda").normal_(generator=gen).to(dtype)
    return out


def prepare(case, seed):
    c, L = case, _lists(case, seed)
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    B, H, D, how, n_q = c["B"], c["H"], c["D"], c["how"], c["n_q"]
    kv = DTYPES[c["dtype"]]
    dt = torch.bfloat16 if c["dtype"] == "fp8" else kv
    s = {"how": how, "n_q": n_q, "ctx": _dev(L["ctx"])}
    i32 = dict(dtype=torch.int32, device="cuda")
    s["status"] = torch.zeros(1, **i32)
    rows = (B, H, n_q, D) if how == "multiq" else (B, H, D)
    s["q"] = _normal(rows, dt, gen)
    s["out"] = torch.zeros(rows, dtype=dt, device="cuda")
    s["lse"] = torch.zeros(rows[:-1], dtype=torch.float32, device="cuda")
    if how == "paged":
        ps = c["page_size"]
        per = (c["ctx"] + ps - 1) // ps
        pages = B * per
        s["k"], s["v"] = (_normal((pages, ps, c["H_kv"], D), kv, gen) for _ in range(2))
        s["table"] = torch.randperm(pages, device="cuda", generator=gen).to(torch.int32).view(B, per)
        s["paging"] = ssa.make_paging(s["table"], ps, pages)
        s["desc"] = ssa.make_desc_paged(s["q"], s["k"], s["v"], s["out"], c["ctx"])
    else:
        s["k"], s["v"] = (_normal((B, c["H_kv"], c["ctx"], D), kv, gen) for _ in range(2))
        if how == "multiq":
            s["desc"], _, s["q_stride_t"], s["o_stride_t"] = ssa.make_desc_multiq(s["q"], s["k"], s["v"], s["out"])
        else:
            s["desc"] = ssa.make_desc(s["q"], s["k"], s["v"], s["out"])
    if how in ("dense", "multiq"):
        s["max_selected"] = c["ctx"]
    else:
        s["max_selected"], s["max_spans"] = L["bound"], L["max_spans"]
        stride = (_most_selected(c) + 31) // 32 * 32
        s["index"], s["counts"] = torch.full((B, stride), -1, **i32), torch.zeros(B, **i32)
    if how == "refs":
        n_lines = [len(x) for x in L["lines"]]
        tables = [_offsets(L["lines"]), _pairs(L["lines"]), np.concatenate([[0], np.cumsum(n_lines)]).astype(np.int32),
                  np.concatenate([np.arange(n) for n in n_lines]).astype(np.int32), _offsets(L["refs"]), _pairs(L["refs"]),
                  np.full(B, c["prefix"], np.int32), np.asarray(L["line_start"], np.int32)]
        s["tables"] = [_dev(t) for t in tables] + [s["ctx"]]
    elif how not in ("dense", "multiq"):
        s["offsets"], s["spans"] = _dev(_offsets(L["spans"])), _dev(_pairs(L["spans"]))
    if how == "blockmask":
        bs = s["block_size"] = c["block_size"]
        cap = (c["ctx"] + bs - 1) // bs
        s["max_blocks"] = (int(L["ctx"].max()) + bs - 1) // bs
        s["block_idx"], s["block_mask"] = torch.full((B, cap), -1, **i32), torch.zeros((B, cap, bs // 32), **i32)
    if how in ("sparse", "paged"):
        ssa.spans_to_index(s["offsets"], s["spans"], s["ctx"], s["index"], s["counts"], s["status"])

    # workspace and plan, kept over the life of a generation
    d = s["desc"]
    need = {"multiq": lambda: ssa.decode_multiq_workspace_bytes(d, n_q, s["max_selected"]),
            "blockmask": lambda: ssa.decode_blockmask_workspace_bytes(d, s["block_size"], s["max_blocks"]),
            "step": lambda: ssa.decode_spans_workspace_bytes(d, s["max_selected"], s["max_spans"]),
            "host_step": lambda: ssa.decode_spans_workspace_bytes(d, s["max_selected"], s["max_spans"]),
            }.get(how, lambda: ssa.decode_workspace_bytes(d, s["max_selected"]))()
    s["workspace"] = torch.empty(max(need, 16), dtype=torch.uint8, device="cuda")
    if how == "step":
        s["step"] = ssa.make_step(s["offsets"], s["spans"], s["ctx"], s["index"], s["counts"], s["q"], s["k"], s["v"],
                                  s["max_selected"], s["out"], s["lse"], s["workspace"], s["status"], max_spans=s["max_spans"])
    elif how == "host_step":
        _host_arenas(s)
    return s


def _host_arenas(s):
    """What changes per step in one device and one pinned host arena; rows and lse land in pinned memory directly."""
    inputs = [s["q"], s["ctx"], s["offsets"], s["spans"]]
    sizes = [(t.numel() * t.element_size() + 255) // 256 * 256 for t in inputs]
    arena = torch.zeros(sum(sizes), dtype=torch.uint8, device="cuda")
    views, at = [], 0
    for t, n in zip(inputs, sizes):
        v = arena[at:at + t.numel() * t.element_size()].view(t.dtype).view(t.shape)
        v.copy_(t)
        views.append(v)
        at += n
    s["q"], s["ctx"], s["offsets"], s["spans"] = views
    s["arena"], s["h_in"] = arena, arena.cpu().pin_memory()
    B = s["ctx"].numel()
    pad = (4 * B + 255) // 256 * 256
    s["d_tail"] = torch.zeros(pad + 256, dtype=torch.uint8, device="cuda")
    s["counts"] = s["d_tail"][:4 * B].view(torch.int32)
    s["status"] = s["d_tail"][pad:pad + 4].view(torch.int32)
    s["h_tail"] = torch.zeros(pad + 256, dtype=torch.uint8).pin_memory()
    s["h_counts"] = s["h_tail"][:4 * B].view(torch.int32)
    s["h_out"], s["h_lse"] = torch.zeros_like(s["out"], device="cpu").pin_memory(), torch.zeros_like(s["lse"], device="cpu").pin_memory()
    s["step"] = ssa.make_step(s["offsets"], s["spans"], s["ctx"], s["index"], s["counts"], s["q"], s["k"], s["v"],
                              s["max_selected"], s["h_out"], s["h_lse"], s["workspace"], s["status"], host_in=s["h_in"],
                              dev_in=s["arena"], host_out=s["h_tail"], dev_out=s["d_tail"], copy_by_kernel=True,
                              max_spans=s["max_spans"])


# ---- one pass ---------------------------------------------------------------------------------------------------
def run(s):
    how = s["how"]
    if how == "step":
        ssa.decode_step(s["desc"], s["step"])
        return s["out"], s["lse"], s["index"], s["counts"]
    if how == "host_step":
        ssa.decode_step(s["desc"], s["step"])
        return s["h_out"], s["h_lse"], s["index"], s["h_counts"]
    if how == "dense":
        ssa.decode_attn_dense(s["desc"], s["q"], s["k"], s["v"], s["ctx"], s["out"], s["lse"], s["workspace"], s["status"])
        return s["out"], s["lse"]
    if how == "multiq":
        ssa.decode_attn_dense_multiq(s["desc"], s["n_q"], s["q_stride_t"], s["o_stride_t"], s["q"], s["k"], s["v"],
                                     s["ctx"], s["out"], s["lse"], s["workspace"], s["status"])
        return s["out"], s["lse"]
    if how == "blockmask":
        ssa.spans_to_blockmask(s["offsets"], s["spans"], s["ctx"], s["block_size"], s["block_idx"], s["block_mask"],
                               s["counts"], s["status"])
        ssa.decode_attn_blockmask(s["desc"], s["q"], s["k"], s["v"], s["ctx"], s["block_idx"], s["block_mask"],
                                  s["counts"], s["block_size"], s["max_blocks"], s["out"], s["lse"], s["workspace"],
                                  s["status"])
        return s["out"], s["lse"], s["block_idx"], s["block_mask"], s["counts"]
    if how == "paged":
        ssa.decode_attn_sparse_paged(s["desc"], s["q"], s["k"], s["v"], s["paging"], s["ctx"], s["index"], s["counts"],
                                     s["max_selected"], s["out"], s["lse"], s["workspace"], s["status"])
        return s["out"], s["lse"]
    if how == "refs":
        ssa.refs_to_index(*s["tables"], s["index"], s["counts"], s["status"])
    ssa.decode_attn_sparse(s["desc"], s["q"], s["k"], s["v"], s["ctx"], s["index"], s["counts"], s["max_selected"],
                           s["out"], s["lse"], s["workspace"], s["status"])
    return (s["out"], s["lse"], s["index"], s["counts"]) if how == "refs" else (s["out"], s["lse"])


def work(case):
    """Selected K and V rows read once, queries read once, rows and lse written once; 4 D operations per selected row
    and query row.  (The lists are a few bytes per row of 16 KB; the counts are those of one seed.)"""
    c = case
    selected = float(_lists(c, 1)["selected"].sum())
    query_rows = c["H"] * c["n_q"]
    return {"bytes": selected * _cache_row_bytes(c) + c["B"] * query_rows * (4.0 * c["D"] + 4.0),
            "flops": 4.0 * c["D"] * selected * query_rows}


def tolerance(case):
    """Rows come in 16 bits (lists are whole numbers and do not differ): against the same attention in 64 bits the
    rounding of the rows alone measures 1.7e-3 (bf16) or 2.1e-4 (f16) in the 2-norm, and at most 2^-8 or 2^-11 of
    a value; about four times that is allowed."""
    if case["dtype"] == "f16":
        return {"rel": 8e-4, "max": 2e-3}
    return {"rel": 6e-3, "max": 1.6e-2}


# ---- the same in 64 bits ----------------------------------------------------------------------------------------
def exact(case, seed):
    """What run() returns for these inputs: softmax(q K^T / sqrt(D)) V over each request's selected positions in
    64 bits, and the lists as they stand."""
    c, L, s = case, _lists(case, seed), prepare(case, seed)
    B, H, D, how = c["B"], c["H"], c["D"], c["how"]
    q = s["q"].double().reshape(B, H * c["n_q"], D)
    group = H * c["n_q"] // c["H_kv"]
    rows, lse, chosen = torch.empty_like(q), torch.empty(q.shape[:2], dtype=torch.float64, device="cuda"), []
    for b in range(B):
        n = int(L["ctx"][b])
        if how in ("dense", "multiq"):
            hit = np.ones(n, bool)
        else:
            hit = np.zeros(n, bool)
            for st, e in _request_spans(c, L, b):
                hit[st:e] = True
        at = np.flatnonzero(hit)
        chosen.append(at)
        pos = _dev(at)
        if how == "paged":
            ps = c["page_size"]
            pool = s["table"][b].long()[pos // ps] * ps + pos % ps
            k, v = (s[t].reshape(-1, c["H_kv"], D)[pool].transpose(0, 1) for t in "kv")
        else:
            k, v = (s[t][b].view(torch.uint8 if s[t].element_size() == 1 else s[t].dtype)[:, pos].view(s[t].dtype) for t in "kv")
        scores = q[b].view(c["H_kv"], group, D) @ k.double().transpose(1, 2) / math.sqrt(D)
        top = torch.logsumexp(scores, -1, keepdim=True)
        rows[b] = (torch.exp(scores - top) @ v.double()).reshape(-1, D)
        lse[b] = top.reshape(-1)
    out = [rows.view(s["out"].shape), lse.view(s["lse"].shape)]
    if how in ("step", "host_step", "refs"):
        index, counts = np.full(tuple(s["index"].shape), -1, np.int32), np.zeros(B, np.int32)
        for b, at in enumerate(chosen):
            index[b, :len(at)], counts[b] = at, len(at)
        out += [index, counts]
    elif how == "blockmask":
        bs = c["block_size"]
        idx = np.full(tuple(s["block_idx"].shape), -1, np.int32)
        mask, counts = np.zeros(tuple(s["block_mask"].shape), np.uint32), np.zeros(B, np.int32)
        for b, at in enumerate(chosen):
            blocks, slot = np.unique(at // bs, return_inverse=True)
            idx[b, :len(blocks)], counts[b] = blocks, len(blocks)
            np.bitwise_or.at(mask[b], (slot, at % bs // 32), (np.uint32(1) << (at % 32).astype(np.uint32)))
        out += [idx, mask.view(np.int32), counts]
    return tuple(out)


def _request_spans(c, L, b):
    if c["how"] != "refs":
        return L["spans"][b]
    named = [ln for lo, hi in L["refs"][b] for ln in L["lines"][b][lo:hi + 1]]
    return [(0, c["prefix"]), (L["line_start"][b], int(L["ctx"][b]))] + named
