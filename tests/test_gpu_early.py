"""What blocks do before the launch in front of theirs has ended: they prefetch by lists, lengths and page tables, cut full contexts
and make lists by what may still be a former step's, or nothing at all.  Results are those of the inputs as the launch in front
leaves them."""
import numpy as np
import pytest
import torch

from oracle import ssa_oracle as O
from paper_2404_09336_b200 import ssa

from gpu_util import DEV

pytestmark = pytest.mark.gpu


def rows_of(q, k, v, index, counts):
    """softmax(q K^T / sqrt(D)) V over the listed rows, in 64 bits."""
    B, H, D = q.shape
    out = torch.zeros(B, H, D, dtype=torch.float64, device=DEV)
    for b in range(B):
        at = index[b, :int(counts[b])].long()
        if len(at) == 0:
            continue
        kb, vb = (x[b][:, at].double().repeat_interleave(H // x.shape[1], 0) for x in (k, v))
        p = torch.softmax(torch.einsum("hd,htd->ht", q[b].double(), kb) / D ** 0.5, -1)
        out[b] = torch.einsum("ht,htd->hd", p, vb)
    return out


# one block more or less than one that prefetches, than fit the chip; lists of one, two turns and a row more
@pytest.mark.parametrize("B,H,Hkv,D,rows,page_size", [
    (74, 8, 8, 128, 65, 0), (75, 8, 8, 128, 129, 0), (47, 8, 8, 128, 200, 0), (37, 32, 32, 64, 257, 0),
    (40, 8, 8, 128, 130, 16), (9, 32, 8, 128, 193, 0), (37, 32, 8, 128, 300, 0), (37, 32, 8, 128, 129, 16)])
@pytest.mark.parametrize("before", [-1, 0x7FFFFFFF, -0x80000000])
def test_lists_of_an_index_launch_in_front(B, H, Hkv, D, rows, page_size, before):
    gen = torch.Generator(device=DEV).manual_seed(B * rows + D)
    T = 1024
    q = torch.randn(B, H, D, device=DEV, generator=gen).bfloat16()
    k, v = (torch.randn(B, Hkv, T, D, device=DEV, generator=gen).bfloat16() for _ in range(2))
    i32 = dict(dtype=torch.int32, device=DEV)
    spans = torch.randint(0, T - rows, (6, B, 2), device=DEV, generator=gen, dtype=torch.int32)
    spans[:, :, 1] = spans[:, :, 0] + torch.randint(1, rows + 1, (6, B), device=DEV, generator=gen, dtype=torch.int32)
    offsets = torch.arange(B + 1, **i32)
    ctx, table = torch.full((B,), before, **i32), None
    kc, vc = k, v
    if page_size:                                        # the same rows through a shuffled page table
        per = T // page_size
        table = torch.randperm(B * per, device=DEV, generator=gen).to(torch.int32).view(B, per)
        kc, vc = (torch.empty(B * per, page_size, Hkv, D, dtype=torch.bfloat16, device=DEV) for _ in range(2))
        for pool, x in ((kc, k), (vc, v)):
            pool[table.long()] = x.view(B, Hkv, per, page_size, D).permute(0, 2, 3, 1, 4)
    index, counts, status = torch.full((B, rows + 7), before, **i32), torch.full((B,), before, **i32), torch.zeros(1, **i32)
    outs = [torch.full((B, H, D), 7.0, device=DEV) for _ in spans]
    desc = ssa.make_desc_paged(q, kc, vc, outs[0], T) if page_size else ssa.make_desc(q, k, v, outs[0])
    ws = torch.empty(max(ssa.decode_workspace_bytes(desc, rows), 16), dtype=torch.uint8, device=DEV)
    full_table = table.clone() if page_size else None
    if page_size:
        table.fill_(before)
    torch.cuda.synchronize()
    ctx.fill_(T)
    if page_size:
        table.copy_(full_table)
        paging = ssa.make_paging(table, page_size, B * (T // page_size))
    lists = []
    for sp, out in zip(spans, outs):                     # (the index launch has ended when attention blocks begin)
        ssa.spans_to_index(offsets, sp, ctx, index, counts, status)
        if page_size:
            ssa.decode_attn_sparse_paged(desc, q, kc, vc, paging, ctx, index, counts, rows, out, None, ws, status)
        else:
            ssa.decode_attn_sparse(desc, q, k, v, ctx, index, counts, rows, out, None, ws, status)
        lists.append((index.clone(), counts.clone()))
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    for sp, out, (idx, cnt) in zip(spans, outs, lists):
        assert torch.equal(cnt, sp[:, 1] - sp[:, 0])
        # fp32 rows: weights exact to 2^-16 (row-sharing kernel) or better, so 1e-4 of values of order 1 is ample
        assert float((out.double() - rows_of(q, k, v, idx, cnt)).abs().max()) < 1e-4


# blocks of one head, of eight and sixteen warps, row-sharing (ordinary, wide, two chunks, above sixteen heads)
@pytest.mark.parametrize("B,H,Hkv,D,dtype", [
    (80, 8, 8, 128, "bf16"), (20, 8, 8, 128, "bf16"), (3, 8, 8, 64, "bf16"), (40, 32, 8, 128, "bf16"), (40, 8, 2, 128, "fp8"),
    (3, 32, 8, 128, "bf16"), (20, 20, 1, 128, "bf16")])
def test_lists_and_spans_that_an_attention_launch_in_front_writes(B, H, Hkv, D, dtype):
    """An attention launch lets the next one's blocks move in as soon as its own have: they then read what it has yet to write.
    Its lists are the next call's: as lists, and their pairs as spans, with its counts as contexts."""
    gen = torch.Generator(device=DEV).manual_seed(B * H + D)
    T, rows = 700, 300
    q = torch.randn(B, H, D, device=DEV, generator=gen).bfloat16()
    kv = torch.float8_e4m3fn if dtype == "fp8" else torch.bfloat16
    k, v = (torch.randn(B, Hkv, T, D, device=DEV, generator=gen).bfloat16().to(kv) for _ in range(2))
    i32 = dict(dtype=torch.int32, device=DEV)
    n = 8
    starts = torch.randint(0, 300, (n, B), device=DEV, generator=gen, dtype=torch.int32)
    lengths = torch.randint(1, rows // 10, (n, B), device=DEV, generator=gen, dtype=torch.int32) * 10
    lengths[0], lengths[1] = 60, 290                     # the same for all, then others everywhere
    spans = torch.stack([starts, starts + lengths], -1).contiguous()
    ctx, offsets = torch.full((B,), T, **i32), torch.arange(B + 1, **i32)
    index, counts = torch.full((B, rows), 5, **i32), torch.zeros(B, **i32)
    pairs = 29                                           # at most 32 are merged by a warp
    status = torch.zeros(1, **i32)
    out = [torch.full((n, B, H, D), 7.0, device=DEV) for _ in range(3)]
    scratch = torch.empty_like(out[0][0])
    desc = ssa.make_desc(q, k, v, scratch)
    ws = torch.empty(max(ssa.decode_spans_workspace_bytes(desc, rows, 150), 16), dtype=torch.uint8, device=DEV)
    table, table_counts = torch.full((B, 2 * pairs), 3, **i32), torch.zeros(B, **i32)
    pair_offsets = torch.arange(B + 1, **i32) * pairs
    index2, counts2 = torch.full((B, pairs), 5, **i32), torch.zeros(B, **i32)
    block_idx, block_mask, counts3 = torch.zeros(B, 24, **i32), torch.zeros(B, 24, 1, **i32), torch.zeros(B, **i32)
    kept, lists, (kr, vr) = [], [], (k.bfloat16(), v.bfloat16())
    torch.cuda.synchronize()
    for i in range(n):
        ssa.decode_attn_spans(desc, q, k, v, ctx, offsets, spans[i], 1, rows, out[0][i], index_out=index, counts_out=counts,
                              workspace=ws, dev_status=status)
        ssa.decode_attn_sparse(desc, q, k, v, ctx, index, counts, rows, out[1][i], None, ws, status)
        # the first pairs of a list of 2 * pairs rows, as a table of spans without offsets
        ssa.decode_attn_spans(desc, q, k, v, ctx, offsets, spans[i], 1, 2 * pairs, out[2][i], index_out=table,
                              counts_out=table_counts, workspace=ws, dev_status=status)
        ssa.decode_attn_spans(desc, q, k, v, counts, None, table, pairs, pairs, out[2][i], workspace=ws, dev_status=status)
        kept.append((index.clone(), counts.clone(), table.clone()))
        # and as span lists of the kernels that make lists of them
        for call, got in ((ssa.spans_to_index, (index2, counts2)), (ssa.spans_to_blockmask, (32, block_idx, block_mask, counts3))):
            ssa.decode_attn_spans(desc, q, k, v, ctx, offsets, spans[i], 1, 2 * pairs, scratch, index_out=table,
                                  counts_out=table_counts, workspace=ws, dev_status=status)
            call(pair_offsets, table.view(-1, 2), counts, *got, status)
        lists.append([x.clone() for x in (index2, counts2, block_idx, block_mask, counts3)])
    torch.cuda.synchronize()
    for i, (idx, cnt, tab) in enumerate(kept):
        assert torch.equal(cnt, lengths[i])
        want = rows_of(q, kr, vr, idx, cnt)
        for got in (out[0][i], out[1][i]):
            assert float((got.double() - want).abs().max()) < 1e-4
        # the pairs of the table are (p, p + 1), or (3, 3) where nothing has been written, below the contexts that the counts are
        at, live = tab[:, 0::2], (tab[:, 1::2] > tab[:, 0::2]) & (tab[:, 0::2] < cnt[:, None])
        chosen, num = torch.zeros(B, pairs, **i32), torch.zeros(B, **i32)
        for b in range(B):
            rows_b = at[b][live[b]].unique()
            chosen[b, :len(rows_b)], num[b] = rows_b, len(rows_b)
            index2, counts2, block_idx, block_mask, counts3 = (x[b] for x in lists[i])
            assert int(counts2) == len(rows_b) and torch.equal(index2[:len(rows_b)], rows_b)
            blocks = (rows_b // 32).unique()
            words = [sum(1 << int(t) % 32 for t in rows_b if int(t) // 32 == int(w)) for w in blocks]
            assert int(counts3) == len(blocks) and torch.equal(block_idx[:len(blocks)], blocks)
            assert [int(w) & 0xFFFFFFFF for w in block_mask[:len(blocks), 0]] == words
        assert float((out[2][i].double() - rows_of(q, kr, vr, chosen, num)).abs().max()) < 1e-4


class Writer:
    """An attention launch that lets the next launch's blocks in as soon as its own have begun, and leaves at its end what that one
    reads: `numbers` int32 (below 0x7c00) in `words`.  Its output rows are fp16; a request's list holds 255 rows whose weight is
    0 and one row of V that is the numbers: each the bits of a value, and a zero for the upper half."""
    ROWS = 256

    def __init__(self, numbers, turns, before):
        heads = -(-numbers // 64)
        assert heads <= 74                               # SMs are left for the next launch's blocks
        half = dict(dtype=torch.float16, device=DEV)
        self.q = torch.ones(1, heads, 128, **half)
        self.k = torch.full((1, heads, turns + self.ROWS - 1, 128), -60.0, **half)
        self.k[:, :, :turns] = 0
        self.v = torch.zeros_like(self.k)
        rows = torch.arange(turns, turns + self.ROWS - 1, dtype=torch.int32, device=DEV)
        self.index = torch.stack([torch.cat([rows, torch.full_like(rows[:1], t)])[None] for t in range(turns)])
        self.count, self.ctx = (torch.full((1,), n, dtype=torch.int32, device=DEV) for n in (self.ROWS, self.k.shape[2]))
        self.out = torch.empty(1, heads, 128, **half)
        self.words = self.out.view(torch.int32).view(-1)
        self.words.fill_(before)
        self.desc = ssa.make_desc(self.q, self.k, self.v, self.out)
        self.ws = torch.empty(ssa.decode_workspace_bytes(self.desc, self.ROWS), dtype=torch.uint8, device=DEV)

    def set(self, turn, numbers):
        """What the launch of that turn leaves."""
        words = np.zeros(len(self.words), np.int32)
        words[:len(numbers)] = numbers
        assert 0 <= words.min() and words.max() < 0x7C00
        self.v[0, :, turn] = torch.from_numpy(words).to(DEV).view(torch.float16).view(-1, 128)

    def write(self, turn):
        ssa.decode_attn_sparse(self.desc, self.q, self.k, self.v, self.ctx, self.index[turn], self.count, self.ROWS, self.out, None,
                               self.ws)


def in_line(turns):
    """The turns, twice: the first time round kernels may have to be loaded, which parts launches.  What is launched meanwhile
    stands in line, and begins as soon as the launch in front lets it."""
    big = torch.empty(2 << 30, dtype=torch.uint8, device=DEV)
    for _ in range(2):
        torch.cuda.synchronize()
        for i in range(3):
            big.fill_(i)
        yield from range(turns)


# rows shared by 4 heads (and tokens), over 8-bit rows, by 20 heads: by two blocks side by side
@pytest.mark.parametrize("B,H,Hkv,T,n_q,dtype", [
    (17, 32, 8, 2560, 1, "bf16"), (17, 16, 8, 2560, 2, "f16"), (17, 32, 8, 2560, 1, "fp8"), (34, 40, 2, 8190, 1, "bf16")])
def test_full_contexts_cut_by_lengths_that_the_launch_in_front_writes(B, H, Hkv, T, n_q, dtype):
    """Full contexts are cut on the device, alike ones otherwise than ragged ones: the lengths change from one to the other."""
    gen, rng = torch.Generator(device=DEV).manual_seed(B + H), np.random.default_rng(T + H)
    tq = torch.float16 if dtype == "f16" else torch.bfloat16
    q = torch.randn(B, H, n_q, 128, device=DEV, generator=gen).to(tq)
    k, v = (torch.randn(B, Hkv, T, 128, device=DEV, generator=gen).to(tq) for _ in range(2))
    if dtype == "fp8":
        k, v = k.to(torch.float8_e4m3fn), v.to(torch.float8_e4m3fn)
    turns = 8
    writer, lengths = Writer(B, turns, 3), []
    for t in range(turns):
        alike, ragged = rng.integers(T - 64, T + 1, B), rng.integers(1, T // 16, B)
        ragged[rng.integers(0, B)] = T
        lengths.append((ragged, alike)[t % 2])
        writer.set(t, lengths[t])
    outs, again = (torch.full((turns, B, H, n_q, 128), 7.0, device=DEV) for _ in range(2))
    desc, *tokens = ssa.make_desc_multiq(q, k, v, outs[0])
    ws = torch.empty(ssa.decode_multiq_workspace_bytes(desc, n_q, T), dtype=torch.uint8, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    for t in in_line(turns):
        writer.write(t)
        ssa.decode_attn_dense_multiq(desc, *tokens, q, k, v, writer.words[:B], outs[t], None, ws, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    everything = torch.arange(T, device=DEV).expand(B, T)
    for t in range(turns):
        ctx = torch.from_numpy(lengths[t].astype(np.int32)).to(DEV)
        ssa.decode_attn_dense_multiq(desc, *tokens, q, k, v, ctx, again[t], None, ws, status)
        torch.cuda.synchronize()
        want = rows_of(q.reshape(B, H * n_q, 128), k.to(tq), v.to(tq), everything, ctx)
        assert float((outs[t].reshape(B, H * n_q, 128).double() - want).abs().max()) < 1e-4, t
        assert torch.equal(outs[t], again[t]), t


GPU_BITS = {O.ST_BAD_SPAN: ssa.DEV_BAD_SPAN, O.ST_CLIPPED: ssa.DEV_CLIPPED, O.ST_OVERFLOW: ssa.DEV_OVERFLOW,
            O.ST_BAD_REF: ssa.DEV_BAD_REF}
LIST_LENGTHS = [0, 1, 5, 30, 31, 32, 33, 64, 100, 255, 256, 257, 300]   # spans: about where the ways to rank them change


def random_spans(rng, n, top):
    starts = rng.integers(0, top, n)
    return np.stack([starts, starts + rng.integers(0, 40, n)], -1)


@pytest.mark.parametrize("before", [-1, 0x7FFFFFFF, 0])
@pytest.mark.parametrize("written", ["offsets", "contexts", "offsets and contexts", "all"])
@pytest.mark.parametrize("block_size", [0, 32, 256])      # 0: index lists; else blocked lists
def test_span_lists_whose_places_the_launch_in_front_writes(block_size, written, before):
    """Offsets, contexts and spans rewritten in place between calls: every block works by what the launch in front leaves."""
    rng = np.random.default_rng(len(written))
    B, T, turns, stride = 13, 3000, 8, 3000
    i32 = dict(dtype=torch.int32, device=DEV)
    n_spans = sum(LIST_LENGTHS) + 20
    turn = []
    for t in range(turns):
        lengths = rng.permutation(LIST_LENGTHS) if t % 3 else rng.permutation(LIST_LENGTHS[:6] + [2] * 7)
        offsets = np.concatenate([[0], np.cumsum(lengths)]) + rng.integers(0, 20)
        turn.append(dict(offsets=offsets, contexts=rng.integers(0, T, B), spans=random_spans(rng, n_spans, T)))
    for x in turn[1:]:
        for name in ("offsets", "contexts", "spans"):
            if name not in written and written != "all":
                x[name] = turn[0][name]
    at = {"offsets": slice(0, B + 1), "contexts": slice(32, 32 + B), "spans": slice(64, 64 + 2 * n_spans)}
    writer = Writer(64 + 2 * n_spans, turns, before)
    for t, x in enumerate(turn):
        words = np.zeros(64 + 2 * n_spans, np.int32)
        for name, where in at.items():
            words[where] = x[name].reshape(-1)
        writer.set(t, words)
    tensors = {name: writer.words[where] if name in written or written == "all" else
               torch.from_numpy(turn[0][name].reshape(-1).astype(np.int32)).to(DEV) for name, where in at.items()}
    counts, status = torch.full((turns, B), -7, **i32), torch.zeros(turns, **i32)
    bs = block_size or 32
    listed = torch.full((turns, B, T // bs + 1 if block_size else stride), -7, **i32)
    masks = torch.full((turns, B, T // bs + 1, bs // 32), -7, **i32)
    args = tensors["offsets"], tensors["spans"], tensors["contexts"]
    for t in in_line(turns):
        writer.write(t)
        if block_size:
            ssa.spans_to_blockmask(*args, bs, listed[t], masks[t], counts[t], status[t:])
        else:
            ssa.spans_to_index(*args, listed[t], counts[t], status[t:])
    torch.cuda.synchronize()
    listed, masks, counts, status = (x.cpu().numpy() for x in (listed, masks, counts, status))
    for t, x in enumerate(turn):
        want_status = 0
        for b in range(B):
            spans, n = x["spans"][x["offsets"][b]:x["offsets"][b + 1]], int(x["contexts"][b])
            want_status |= O.spans_status(spans, n, stride)
            want, words = O.spans_to_blockmask(spans, n, bs) if block_size else (O.spans_to_index(spans, n), None)
            assert counts[t, b] == len(want) and listed[t, b, :len(want)].tolist() == want.tolist(), (t, b)
            assert np.all(listed[t, b, len(want):] == -7)
            if block_size:
                assert np.array_equal(masks[t, b, :len(want)].view(np.uint32), words), (t, b)
        assert status[t] == sum(v for k, v in GPU_BITS.items() if want_status & k)


@pytest.mark.parametrize("before", [-1, 0x7FFFFFFF])
@pytest.mark.parametrize("written", [
    "line_offsets", "lines", "anchor_offsets", "anchors", "ref_offsets", "refs", "prefix", "start", "ctx", "all"])
def test_references_whose_tables_the_launch_in_front_writes(written, before):
    """Every table of ssa_refs_to_index, and all of them, rewritten in place between calls."""
    rng = np.random.default_rng(len(written))
    B, turns, stride, T = 9, 8, 3000, 3000
    i32 = dict(dtype=torch.int32, device=DEV)
    at, end = {}, 0
    for name, size in dict(line_offsets=B + 1, anchor_offsets=B + 1, ref_offsets=B + 1, prefix=B, start=B, ctx=B, lines=1800,
                           anchors=1400, refs=700).items():
        at[name], end = slice(end, end + size), end + size + size % 2          # (pairs stay on 8 bytes)
    turn = []
    for t in range(turns):
        n_lines, n_anchors = rng.choice([0, 20, 60, 90], B), rng.choice([1, 40, 150], B)
        n_refs = rng.choice([0, 1, 2, 31, 33], B)
        if t == turns - 2:
            n_lines[0], n_anchors[1], n_refs[2] = 100, 560, 40                 # a table that is not copied
            n_lines[1:], n_anchors[2:] = 60, 40
        place = lambda n: np.concatenate([[0], np.cumsum(n)]) + 2
        lo = rng.integers(0, 140, 350)
        turn.append(dict(
            line_offsets=place(n_lines), anchor_offsets=place(n_anchors), ref_offsets=place(n_refs),
            prefix=rng.integers(0, 80, B), start=rng.integers(T - 200, T, B), ctx=rng.integers(T // 2, T, B),
            lines=random_spans(rng, 900, T), anchors=rng.integers(0, 100, 1400),
            refs=np.stack([lo, lo + rng.integers(0, 12, 350)], -1)))
    for x in turn[1:]:
        for name in at:
            if written not in (name, "all"):
                x[name] = turn[0][name]
    writer = Writer(end, turns, before)
    for t, x in enumerate(turn):
        words = np.zeros(end, np.int32)
        for name, where in at.items():
            words[where] = x[name].reshape(-1)
        writer.set(t, words)
    tables = [writer.words[where] if written in (name, "all") else
              torch.from_numpy(turn[0][name].reshape(-1).astype(np.int32)).to(DEV)
              for name, where in ((n, at[n]) for n in ("line_offsets", "lines", "anchor_offsets", "anchors", "ref_offsets", "refs",
                                                       "prefix", "start", "ctx"))]
    listed, counts = torch.full((turns, B, stride), -7, **i32), torch.full((turns, B), -7, **i32)
    status = torch.zeros(turns, **i32)
    for t in in_line(turns):
        writer.write(t)
        ssa.refs_to_index(*tables, listed[t], counts[t], status[t:])
    torch.cuda.synchronize()
    listed, counts, status = listed.cpu().numpy(), counts.cpu().numpy(), status.cpu().numpy()
    for t, x in enumerate(turn):
        want_status = 0
        for b in range(B):
            own = lambda name, offsets: x[name][x[offsets][b]:x[offsets][b + 1]]
            spans, bits = O.resolve_references(own("lines", "line_offsets"), own("anchors", "anchor_offsets"),
                                               own("refs", "ref_offsets"), x["prefix"][b], x["start"][b], x["ctx"][b])
            assert len(spans) <= 2048
            want_status |= bits | O.spans_status(spans, x["ctx"][b], stride)
            rows = O.spans_to_index(spans, x["ctx"][b])
            assert counts[t, b] == len(rows) and listed[t, b, :len(rows)].tolist() == rows.tolist(), (t, b)
            assert np.all(listed[t, b, len(rows):] == -7)
        assert status[t] == sum(v for k, v in GPU_BITS.items() if want_status & k)


# blocks of one head, of eight and sixteen warps, row-sharing (ordinary, two chunks, 8-bit rows, above sixteen heads)
# and large blocks on both sides of the line for merging early: rows and spans a request may have
@pytest.mark.parametrize("B,H,Hkv,D,dtype,most,cap", [
    (40, 8, 8, 128, "bf16", 900, 30), (20, 8, 8, 128, "f16", 900, 30), (3, 8, 8, 64, "bf16", 900, 30),
    (40, 32, 8, 128, "bf16", 900, 30), (3, 32, 8, 128, "bf16", 900, 30), (40, 8, 2, 128, "fp8", 900, 30),
    (20, 20, 1, 128, "bf16", 900, 30), (20, 8, 8, 128, "bf16", 384, 16), (20, 8, 8, 128, "bf16", 385, 16),
    (10, 8, 8, 128, "f16", 900, 16), (10, 8, 8, 128, "f16", 900, 17)])
@pytest.mark.parametrize("before", [-1, 0])
def test_attention_over_spans_whose_places_the_launch_in_front_writes(B, H, Hkv, D, dtype, most, cap, before):
    """Offsets, contexts and spans of ssa_decode_attn_spans rewritten in place between calls."""
    gen, rng = torch.Generator(device=DEV).manual_seed(B * H + D), np.random.default_rng(B)
    T, turns = 900, 8
    tq = torch.float16 if dtype == "f16" else torch.bfloat16
    q = torch.randn(B, H, D, device=DEV, generator=gen).to(tq)
    k, v = (torch.randn(B, Hkv, T, D, device=DEV, generator=gen).to(tq) for _ in range(2))
    if dtype == "fp8":
        k, v = k.to(torch.float8_e4m3fn), v.to(torch.float8_e4m3fn)
    n_spans = 18 * B + 40
    ends = 3 * B + 1 + (3 * B + 1) % 2                   # (spans lie on 8 bytes)
    writer, turn = Writer(ends + 2 * n_spans, turns, before), []
    for t in range(turns):
        lengths = np.minimum(rng.choice([0, 1, 3, 14, cap], B), min(18, cap) if t % 2 else cap)
        while lengths.sum() > n_spans - 20:
            lengths[rng.integers(B)] = 1
        offsets, spans = np.concatenate([[0], np.cumsum(lengths)]) + rng.integers(0, 20), random_spans(rng, n_spans, T - 40)
        ctx = rng.integers(1, T + 1, B)
        turn.append((offsets, spans, ctx))
        words = np.zeros(ends + 2 * n_spans, np.int32)
        words[:B + 1], words[2 * B:3 * B], words[ends:] = offsets, ctx, spans.reshape(-1)
        writer.set(t, words)
    i32 = dict(dtype=torch.int32, device=DEV)
    outs, status = torch.full((turns, B, H, D), 7.0, device=DEV), torch.zeros(1, **i32)
    listed, counts = torch.full((turns, B, most), -7, **i32), torch.full((turns, B), -7, **i32)
    desc = ssa.make_desc(q, k, v, outs[0])
    ws = torch.empty(max(ssa.decode_spans_workspace_bytes(desc, most, cap), 16), dtype=torch.uint8, device=DEV)
    for t in in_line(turns):
        writer.write(t)
        ssa.decode_attn_spans(desc, q, k, v, writer.words[2 * B:3 * B], writer.words[:B + 1], writer.words[ends:], cap, most, outs[t],
                              index_out=listed[t], counts_out=counts[t], workspace=ws, dev_status=status)
    torch.cuda.synchronize()
    got_lists, got_counts = listed.cpu().numpy(), counts.cpu().numpy()
    for t, (offsets, spans, ctx) in enumerate(turn):
        for b in range(B):
            rows = O.spans_to_index(spans[offsets[b]:offsets[b + 1]], int(ctx[b]))[:most]
            assert got_counts[t, b] == len(rows) and got_lists[t, b, :len(rows)].tolist() == rows.tolist(), (t, b)
        want = rows_of(q, k.to(tq), v.to(tq), listed[t], counts[t])
        assert float((outs[t].double() - want).abs().max()) < 1e-4, t


# one head per block, rows shared by four heads; contiguous and paged
@pytest.mark.parametrize("B,H,Hkv,D,rows,page_size", [
    (24, 32, 32, 128, 150, 0), (24, 32, 32, 64, 150, 0), (24, 32, 8, 128, 150, 0), (24, 32, 32, 128, 120, 16),
    (12, 32, 8, 128, 300, 16)])
@pytest.mark.parametrize("before", [-1, 0x7FFFFFFF, -0x80000000])
def test_lists_that_an_attention_launch_in_front_writes(B, H, Hkv, D, rows, page_size, before):
    """Lists, counts, contexts and page tables rewritten in place between calls over lists and over full contexts."""
    gen, rng = torch.Generator(device=DEV).manual_seed(B * rows + D), np.random.default_rng(D)
    T, turns = 1024, 4
    per = T // page_size if page_size else 0
    q = torch.randn(B, H, D, device=DEV, generator=gen).bfloat16()
    shape = (B * per, page_size, Hkv, D) if page_size else (B, Hkv, T, D)
    k, v = (torch.randn(shape, device=DEV, generator=gen).bfloat16() for _ in range(2))
    at, end = {}, 0
    for name, size in dict(ctx=B, counts=B, index=B * rows, table=B * per).items():
        at[name], end = slice(end, end + size), end + size
    writer, turn = Writer(end, turns, before), []
    for t in range(turns):
        ctx, counts = rng.integers(rows, T + 1, B), rng.integers(0, rows + 1, B)
        index = np.stack([rng.permutation(n)[:rows] for n in ctx])
        turn.append(dict(ctx=ctx, counts=counts, index=index, table=rng.permutation(B * per)))
        writer.set(t, np.concatenate([turn[t][name].reshape(-1) for name in at]))
    ctx, counts, index, table = (writer.words[where] for where in at.values())
    index = index.view(B, rows)
    outs, status = torch.full((2, turns, B, H, D), 7.0, device=DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
    desc = ssa.make_desc_paged(q, k, v, outs[0, 0], T) if page_size else ssa.make_desc(q, k, v, outs[0, 0])
    ws = torch.empty(max(ssa.decode_workspace_bytes(desc, n) for n in (rows, T)), dtype=torch.uint8, device=DEV)
    paging = ssa.make_paging(table.view(B, per), page_size, B * per) if page_size else None
    for t in in_line(turns):
        writer.write(t)
        if page_size:
            ssa.decode_attn_sparse_paged(desc, q, k, v, paging, ctx, index, counts, rows, outs[0, t], None, ws, status)
        else:
            ssa.decode_attn_sparse(desc, q, k, v, ctx, index, counts, rows, outs[0, t], None, ws, status)
        t = (t + 1) % turns                              # other words again
        writer.write(t)
        if page_size:
            ssa.decode_attn_dense_paged(desc, q, k, v, paging, ctx, outs[1, t], None, ws, status)
        else:
            ssa.decode_attn_dense(desc, q, k, v, ctx, outs[1, t], None, ws, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    everything = torch.arange(T, device=DEV).expand(B, T)
    for t, x in enumerate(turn):
        x = {name: torch.from_numpy(a).to(DEV) for name, a in x.items()}
        kc, vc = k, v
        if page_size:                                    # the requests' rows in order
            kc, vc = (pool[x["table"].view(B, per)].reshape(B, T, Hkv, D).transpose(1, 2) for pool in (k, v))
        for out, idx, n in ((outs[0, t], x["index"], x["counts"]), (outs[1, t], everything, x["ctx"])):
            assert float((out.double() - rows_of(q, kc, vc, idx, n)).abs().max()) < 1e-4, t
