"""8-bit (e4m3) cache storage: the attention calls over a cache of uint8 patterns against the fp64 oracle, whose
decoder is written from the format's definition.  Queries are bf16; outputs fp32 or bf16."""
import numpy as np
import pytest
import torch

from oracle import ssa_oracle as O
from paper_2404_09336_b200 import ssa
from paper_2404_09336_b200.inputs import round_to_storage

from gpu_util import DEV
from parity import assert_parity

pytestmark = pytest.mark.gpu


def to_e4m3_bits(x32):
    return torch.from_numpy(np.ascontiguousarray(x32, np.float32)).to(torch.float8_e4m3fn).view(torch.uint8).numpy()


class Fp8Problem:
    def __init__(self, B, H, Hkv, T, D, seed, layout="bhtd"):
        rng = np.random.default_rng(seed)
        self.B, self.H, self.Hkv, self.T, self.D = B, H, Hkv, T, D
        self.q_bits = round_to_storage(rng.standard_normal((B, H, D), dtype=np.float32), "bf16")
        self.k_bits = to_e4m3_bits(rng.standard_normal((B, Hkv, T, D), dtype=np.float32))
        self.v_bits = to_e4m3_bits(rng.standard_normal((B, Hkv, T, D), dtype=np.float32))
        self.q = torch.from_numpy(self.q_bits.view(np.int16)).view(torch.bfloat16).to(DEV)
        k = torch.from_numpy(self.k_bits).view(torch.float8_e4m3fn)
        v = torch.from_numpy(self.v_bits).view(torch.float8_e4m3fn)
        if layout == "bthd":
            self.k = k.permute(0, 2, 1, 3).contiguous().to(DEV).permute(0, 2, 1, 3)
            self.v = v.permute(0, 2, 1, 3).contiguous().to(DEV).permute(0, 2, 1, 3)
        else:
            self.k, self.v = k.to(DEV), v.to(DEV)

    def oracle_kv(self):
        g = self.H // self.Hkv
        return np.repeat(self.k_bits, g, axis=1), np.repeat(self.v_bits, g, axis=1)


@pytest.mark.parametrize("H,Hkv,D,layout,out_dtype", [
    (4, 4, 128, "bhtd", torch.float32), (3, 3, 64, "bthd", torch.float32), (8, 2, 128, "bhtd", torch.bfloat16),
    (2, 2, 128, "bthd", torch.bfloat16)])
def test_sparse_dense_and_span_calls_against_the_oracle(H, Hkv, D, layout, out_dtype):
    B, T = 3, 2000
    p = Fp8Problem(B, H, Hkv, T, D, seed=11 * H + D, layout=layout)
    ctx = [2000, 1333, 300]
    spans = [[(0, 64), (700, 1500), (1990, 2000)], [(5, 9), (100, 130), (1300, 1333), (128, 140)], [(17, 18)]]
    counts, index = [], np.full((B, 1024), -1, np.int32)
    for b in range(B):
        idx = O.spans_to_index(spans[b], ctx[b])
        index[b, :len(idx)] = idx
        counts.append(len(idx))
    d_idx, d_cnt = torch.from_numpy(index).to(DEV), torch.tensor(counts, dtype=torch.int32, device=DEV)
    d_ctx = torch.tensor(ctx, dtype=torch.int32, device=DEV)
    out = torch.full((B, H, D), 7.0, dtype=out_dtype, device=DEV)
    lse = torch.full((B, H), 7.0, dtype=torch.float32, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    desc = ssa.make_desc(p.q, p.k, p.v, out)
    assert desc.kv_dtype == ssa.FP8_E4M3
    ws = torch.empty(max(ssa.decode_workspace_bytes(desc, T), ssa.decode_spans_workspace_bytes(desc, 1024, 8)),
                     dtype=torch.uint8, device=DEV)
    ko, vo = p.oracle_kv()
    native = out_dtype != torch.float32
    scale = 1 / np.sqrt(D)
    ref, ref_lse = O.decode_attn_sparse(p.q_bits, ko, vo, ctx, index, counts, scale, "bf16/e4m3")

    ssa.decode_attn_sparse(desc, p.q, p.k, p.v, d_ctx, d_idx, d_cnt, 1024, out, lse, ws, status)
    torch.cuda.synchronize()
    assert_parity(out.double().cpu().numpy(), ref, native, "index lists over an 8-bit cache")
    np.testing.assert_allclose(lse.double().cpu().numpy(), ref_lse, rtol=1e-5, atol=1e-5)

    out.fill_(7.0)
    offs = torch.tensor(np.cumsum([0] + [len(s) for s in spans]), dtype=torch.int32, device=DEV)
    flat = torch.tensor([x for s in spans for x in s], dtype=torch.int32, device=DEV)
    ssa.decode_attn_spans(desc, p.q, p.k, p.v, d_ctx, offs, flat, 4, 1024, out, lse, None, None, ws, status)
    torch.cuda.synchronize()
    assert_parity(out.double().cpu().numpy(), ref, native, "span lists over an 8-bit cache")

    ssa.decode_attn_dense(desc, p.q, p.k, p.v, d_ctx, out, lse, ws, status)
    torch.cuda.synchronize()
    refd, refd_lse = O.decode_attn_dense(p.q_bits, ko, vo, ctx, scale, "bf16/e4m3")
    assert_parity(out.double().cpu().numpy(), refd, native, "full context over an 8-bit cache")
    np.testing.assert_allclose(lse.double().cpu().numpy(), refd_lse, rtol=1e-5, atol=1e-5)
    assert int(status.item()) == 0


def test_every_e4m3_pattern_is_read_exactly():
    """One selected row per head holding all finite patterns: the output row is that V row, exactly."""
    B, H, T, D = 1, 2, 32, 128
    p = Fp8Problem(B, H, H, T, D, seed=1)
    pats = np.array([x for x in range(256) if x not in (0x7F, 0xFF)], np.uint8)
    v = p.v_bits.copy()
    v[0, 0, 5], v[0, 1, 5] = pats[:128], pats[126:254]
    p.v = torch.from_numpy(v).view(torch.float8_e4m3fn).to(DEV)
    out = torch.zeros((B, H, D), dtype=torch.float32, device=DEV)
    desc = ssa.make_desc(p.q, p.k, p.v, out)
    ws = torch.empty(ssa.decode_workspace_bytes(desc, 32), dtype=torch.uint8, device=DEV)
    idx = torch.full((1, 32), 5, dtype=torch.int32, device=DEV)
    ssa.decode_attn_sparse(desc, p.q, p.k, p.v, torch.tensor([T], dtype=torch.int32, device=DEV), idx,
                           torch.tensor([1], dtype=torch.int32, device=DEV), 32, out, None, ws, None)
    torch.cuda.synchronize()
    want = O.decode_e4m3(v[0, :, 5])
    assert np.array_equal(out.double().cpu().numpy()[0], want)


def test_descriptor_checks():
    p = Fp8Problem(1, 2, 2, 64, 128, seed=2)
    out16 = torch.zeros((1, 2, 128), dtype=torch.float16, device=DEV)
    desc = ssa.make_desc(p.q, p.k, p.v, out16)                  # fp16 output with an 8-bit cache: not offered
    assert ssa.decode_workspace_bytes(desc, 64) == 0
    out = torch.zeros((1, 2, 128), dtype=torch.float32, device=DEV)
    desc = ssa.make_desc(p.q, p.k, p.v, out)
    assert ssa.decode_workspace_bytes(desc, 64) > 0
    desc.k_stride_t = 136                                       # 136 bytes: not a multiple of 16
    assert ssa.decode_workspace_bytes(desc, 64) == 0


@pytest.mark.parametrize("B,group,T,counts", [
    (3, 2, 140, [1, 16, 129]),          # small launches: one head per block ...
    (2, 7, 1100, [1023, 1025]), (3, 8, 700, [15, 17, 700]), (3, 9, 700, [127, 128, 0]), (2, 16, 2600, [2600, 513]),
    (3, 2, 7000, [1, 16, 129]),         # ... and shared rows: list ends around a 16-row tile and a round of the block's tiles
    (3, 8, 7000, [15, 17, 6000]),
    (3, 9, 7000, [127, 128, 0]),        # two head tiles, the second with one head; an empty list
    (3, 16, 7000, [6000, 513, 1]),
    (40, 4, 300, None),                 # one unit for most SMs: the large blocks, index and span lists ...
    (40, 7, 1100, [1023, 1024, 1025, 16, 17] * 8),   # ... list ends around the staging window; a head of the tile missing
    (40, 12, 300, None), (40, 16, 1100, [1025, 1023, 1100, 0] * 10),
    (3, 2, 51000, [51000, 1, 20000]),   # full contexts cut on the device ...
    (3, 16, 51000, [51000, 1, 20000]),  # ... by two-warp teams
])
def test_grouped_heads_over_an_8_bit_cache(B, group, T, counts):
    # fp32 output: weights carry 22 bits or an absolute 2^-37, sums are fp32 over at most 51000 rows: 2^-22 per weight
    # and 2^-24 sqrt(51000) = 1.4e-5 relative per sum bound the error of an N(0, 1) average by 1.5e-5; 2e-5 is asserted.
    # Errors that are independent from row to row average out: in the 2-norm an error of 2^-22 per weight or product
    # stays below 2.4e-7 of the result (measured: at most 2.4e-7, one head per block 2.7e-7); four times that is asserted.
    Hkv, D = 2, 128
    H = group * Hkv
    p = Fp8Problem(B, H, Hkv, T, D, seed=100 * group + T)
    rng = np.random.default_rng(T)
    ctx = [T] * B
    counts = counts or [int(x) for x in rng.integers(1, T + 1, size=B)]
    index = np.full((B, T), -1, np.int32)
    for b, c in enumerate(counts):
        index[b, :c] = np.sort(rng.choice(T, c, replace=False))
    out = torch.full((B, H, D), 7.0, dtype=torch.float32, device=DEV)
    lse = torch.full((B, H), 7.0, dtype=torch.float32, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    d_ctx = torch.tensor(ctx, dtype=torch.int32, device=DEV)
    desc = ssa.make_desc(p.q, p.k, p.v, out)
    # (a full context is cut on the device only in a workspace of its own bound)
    ws = torch.empty(max(ssa.decode_spans_workspace_bytes(desc, T, 4), ssa.decode_workspace_bytes(desc, T)),
                     dtype=torch.uint8, device=DEV)
    ko, vo = p.oracle_kv()

    def check(ref, ref_lse, what):
        torch.cuda.synchronize()
        diff = out.double().cpu().numpy() - ref
        assert float(np.abs(diff).max()) <= 2e-5, what
        assert float(np.linalg.norm(diff)) <= 1e-6 * float(np.linalg.norm(ref)), what
        ok = np.isfinite(ref_lse)
        np.testing.assert_allclose(lse.double().cpu().numpy()[ok], ref_lse[ok], rtol=2e-6, atol=2e-6, err_msg=what)
        assert int(status.item()) == 0

    ssa.decode_attn_sparse(desc, p.q, p.k, p.v, d_ctx, torch.from_numpy(index).to(DEV),
                           torch.tensor(counts, dtype=torch.int32, device=DEV), T, out, lse, ws, status)
    check(*O.decode_attn_sparse(p.q_bits, ko, vo, ctx, index, counts, 1 / np.sqrt(D), "bf16/e4m3"), "index lists")
    ssa.decode_attn_dense(desc, p.q, p.k, p.v, d_ctx, out, lse, ws, status)
    dense = O.decode_attn_dense(p.q_bits, ko, vo, ctx, 1 / np.sqrt(D), "bf16/e4m3")
    check(*dense, "full context")
    ragged = [T // 64 + 64 * (b % 3) if b else T for b in range(B)]
    ssa.decode_attn_dense(desc, p.q, p.k, p.v, torch.tensor(ragged, dtype=torch.int32, device=DEV), out, lse, ws, status)
    check(*O.decode_attn_dense(p.q_bits, ko, vo, ragged, 1 / np.sqrt(D), "bf16/e4m3"), "ragged full contexts")
    flat = torch.tensor([[0, T // 2], [T // 2, T]] * B, dtype=torch.int32, device=DEV)
    offs = torch.arange(0, 2 * B + 1, 2, dtype=torch.int32, device=DEV)
    ssa.decode_attn_spans(desc, p.q, p.k, p.v, d_ctx, offs, flat, 4, T, out, lse, None, None, ws, status)
    check(*dense, "span lists")


@pytest.mark.parametrize("group,rows", [(4, 32), (12, 32), (4, 7000), (12, 7000)])   # one head per block / shared rows
def test_grouped_heads_read_every_e4m3_pattern_exactly(group, rows):
    """One selected row per K/V head: every head of the group returns that V row, exactly; a NaN in K or V shows.  The
    launch is sized for lists of up to `rows`."""
    B, Hkv, T, D = 1, 2, 32, 128
    H = group * Hkv
    p = Fp8Problem(B, H, Hkv, T, D, seed=3)
    pats = np.array([x for x in range(256) if x not in (0x7F, 0xFF)], np.uint8)
    v = p.v_bits.copy()
    v[0, 0, 5], v[0, 1, 5] = pats[:128], pats[126:254]
    out = torch.zeros((B, H, D), dtype=torch.float32, device=DEV)
    desc = ssa.make_desc(p.q, p.k, p.v, out)
    ws = torch.empty(ssa.decode_workspace_bytes(desc, rows), dtype=torch.uint8, device=DEV)
    idx = torch.full((1, rows), 5, dtype=torch.int32, device=DEV)
    one, ctx = (torch.tensor([x], dtype=torch.int32, device=DEV) for x in (1, T))

    def run(v_bits, k=p.k):
        pv = torch.from_numpy(v_bits).view(torch.float8_e4m3fn).to(DEV)
        ssa.decode_attn_sparse(desc, p.q, k, pv, ctx, idx, one, rows, out, None, ws, None)
        torch.cuda.synchronize()
        return out.double().cpu().numpy()[0]

    want = np.repeat(O.decode_e4m3(v[0, :, 5]), group, axis=0)
    assert np.array_equal(run(v), want)
    v[0, 0, 5, 77] = 0x7F
    got = run(v)
    assert np.isnan(got[:group, 77]).all() and np.isfinite(np.delete(got, 77, axis=1)).all()
    v[0, 0, 5, 77] = 0
    k_bits = p.k_bits.copy()
    k_bits[0, 1, 5, 3] = 0xFF
    got = run(v, torch.from_numpy(k_bits).view(torch.float8_e4m3fn).to(DEV))
    assert np.isnan(got[group:]).all() and np.isfinite(got[:group]).all()


@pytest.mark.parametrize("B,group,T,page_size", [(2, 4, 600, 16), (3, 4, 7000, 64), (3, 12, 7000, 16), (40, 12, 300, 32)])
def test_grouped_heads_over_a_paged_8_bit_cache(B, group, T, page_size):
    """The same rows through a page table: index lists bit for bit as from the contiguous cache, full contexts (which the
    contiguous call may cut elsewhere) within the bound of the test above."""
    Hkv, D = 2, 128
    H = group * Hkv
    p = Fp8Problem(B, H, Hkv, T, D, seed=group + T)
    rng = np.random.default_rng(page_size)
    per = (T + page_size - 1) // page_size
    n_pages = B * per + 3
    table = rng.permutation(n_pages)[: B * per].astype(np.int32).reshape(B, per)

    def pool(bits):
        padded = np.zeros((B, per * page_size, Hkv, D), np.uint8)
        padded[:, :T] = bits.transpose(0, 2, 1, 3)
        out = np.full((n_pages, page_size, Hkv, D), 0x7F, np.uint8)         # pages of nobody hold NaN
        out[table.reshape(-1)] = padded.reshape(B * per, page_size, Hkv, D)
        return torch.from_numpy(out).view(torch.float8_e4m3fn).to(DEV)

    kp, vp, d_tab = pool(p.k_bits), pool(p.v_bits), torch.from_numpy(table).to(DEV)
    ctx = [T - 7 * b for b in range(B)]
    counts = [int(x) for x in rng.integers(0, np.asarray(ctx) + 1)]
    index = np.full((B, T), -1, np.int32)
    for b, c in enumerate(counts):
        index[b, :c] = np.sort(rng.choice(ctx[b], c, replace=False))
    d_ctx, d_cnt = (torch.tensor(x, dtype=torch.int32, device=DEV) for x in (ctx, counts))
    d_idx = torch.from_numpy(index).to(DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    got = {}
    for paged in (False, True):
        out = torch.full((B, H, D), 7.0, dtype=torch.float32, device=DEV)
        lse = torch.full((B, H), 7.0, dtype=torch.float32, device=DEV)
        desc = ssa.make_desc_paged(p.q, kp, vp, out, T) if paged else ssa.make_desc(p.q, p.k, p.v, out)
        ws = torch.empty(ssa.decode_workspace_bytes(desc, T), dtype=torch.uint8, device=DEV)
        if paged:
            pg = ssa.make_paging(d_tab, page_size, n_pages)
            ssa.decode_attn_sparse_paged(desc, p.q, kp, vp, pg, d_ctx, d_idx, d_cnt, T, out, lse, ws, status)
        else:
            ssa.decode_attn_sparse(desc, p.q, p.k, p.v, d_ctx, d_idx, d_cnt, T, out, lse, ws, status)
        torch.cuda.synchronize()
        got[paged] = out.cpu().numpy(), lse.cpu().numpy()
    assert all(np.array_equal(x, y) for x, y in zip(got[False], got[True]))
    ssa.decode_attn_dense_paged(desc, p.q, kp, vp, pg, d_ctx, out, lse, ws, status)
    torch.cuda.synchronize()
    ko, vo = p.oracle_kv()
    ref, ref_lse = O.decode_attn_dense(p.q_bits, ko, vo, ctx, 1 / np.sqrt(D), "bf16/e4m3")
    diff = out.double().cpu().numpy() - ref
    assert float(np.linalg.norm(diff)) <= 1e-6 * float(np.linalg.norm(ref))
    np.testing.assert_allclose(lse.double().cpu().numpy(), ref_lse, rtol=2e-6, atol=2e-6)
    assert int(status.item()) == 0


@pytest.mark.parametrize("B,Hkv,sel", [(1, 2, 820), (8, 2, 500), (1, 8, 160)])
def test_small_grouped_launches_one_head_per_block_or_in_the_workspace_of_shared_rows(B, Hkv, sel):
    """Both plans of a small launch: with the workspace of the query, and with one that only holds shared rows (whose
    partial results can be fewer).  Bounds as in the tests above."""
    H, T, D = 32, 1000, 128
    p = Fp8Problem(B, H, Hkv, T, D, seed=sel)
    rng = np.random.default_rng(B)
    index = np.stack([np.sort(rng.choice(T, sel, replace=False)) for _ in range(B)]).astype(np.int32)
    counts = [sel - 3 * b for b in range(B)]
    d_ctx, d_cnt = (torch.tensor(x, dtype=torch.int32, device=DEV) for x in ([T] * B, counts))
    ko, vo = p.oracle_kv()
    ref, ref_lse = O.decode_attn_sparse(p.q_bits, ko, vo, [T] * B, index, counts, 1 / np.sqrt(D), "bf16/e4m3")
    out = torch.full((B, H, D), 7.0, dtype=torch.float32, device=DEV)
    lse = torch.full((B, H), 7.0, dtype=torch.float32, device=DEV)
    desc = ssa.make_desc(p.q, p.k, p.v, out)
    units = B * Hkv
    chunks = min(2 * torch.cuda.get_device_properties(DEV).multi_processor_count // units, -(-sel // 256))
    shared = sum((B * H * chunks * n + 255) // 256 * 256 for n in (4 * D, 8))
    for nbytes in (ssa.decode_workspace_bytes(desc, sel), shared):
        ws = torch.full((nbytes + 4096,), 0xA5, dtype=torch.uint8, device=DEV)
        out.fill_(7.0)
        ssa.decode_attn_sparse(desc, p.q, p.k, p.v, d_ctx, torch.from_numpy(index).to(DEV), d_cnt, sel, out, lse,
                               ws[:nbytes], None)
        torch.cuda.synchronize()
        assert bool((ws[nbytes:] == 0xA5).all())
        assert float(np.linalg.norm(out.double().cpu().numpy() - ref)) <= 1e-6 * float(np.linalg.norm(ref))
        np.testing.assert_allclose(lse.double().cpu().numpy(), ref_lse, rtol=2e-6, atol=2e-6)
    # the same rows as one-token spans, more than a block merges on chip: lists and partial results share the workspace
    spans = np.concatenate([np.stack([r, r + 1], 1)[:c] for r, c in zip(index, counts)]).astype(np.int32)
    offs = torch.from_numpy(np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)).to(DEV)
    nbytes = ssa.decode_spans_workspace_bytes(desc, sel, sel)
    ws2 = torch.full((nbytes + 4096,), 0xA5, dtype=torch.uint8, device=DEV)
    listed = out.clone()
    ssa.decode_attn_sparse(desc, p.q, p.k, p.v, d_ctx, torch.from_numpy(index).to(DEV), d_cnt, sel, listed, lse,
                           torch.empty(ssa.decode_workspace_bytes(desc, sel), dtype=torch.uint8, device=DEV), None)
    ssa.decode_attn_spans(desc, p.q, p.k, p.v, d_ctx, offs, torch.from_numpy(spans).to(DEV), sel, sel, out, lse, None, None,
                          ws2[:nbytes], None)
    torch.cuda.synchronize()
    assert torch.equal(out, listed) and bool((ws2[nbytes:] == 0xA5).all())
    before = ssa.launch_count()                                 # one head per block needs no second pass up to 512 rows
    ssa.decode_attn_sparse(desc, p.q, p.k, p.v, d_ctx, torch.from_numpy(index).to(DEV), d_cnt, sel, out, lse, ws, None)
    assert ssa.launch_count() - before == (2 if sel > 512 else 1)
    torch.cuda.synchronize()


@pytest.mark.parametrize("group", [2, 8, 12, 20])
@pytest.mark.parametrize("kind", ["wide", "tiny", "huge", "spread", "not finite"])
def test_shared_rows_over_an_8_bit_cache_whatever_the_magnitude_of_the_queries(group, kind):
    """The row-sharing kernel scales query rows by powers of two.  Rows near the ends of the bf16 range (with a softmax scale
    that brings the scores back), rows whose elements span 2^40, and rows with an infinity or a NaN next to ordinary ones.
    Bound: scores of up to 8 sqrt(128) |k| carry 2^-24 sqrt(128) relative each; 4e-6 in the 2-norm is asserted (measured at
    most 6.4e-7, the same with unscaled queries)."""
    B, Hkv, T, D = 2, 2, 8000, 128
    H = group * Hkv
    p = Fp8Problem(B, H, Hkv, T, D, seed=group)
    rng = np.random.default_rng(group)
    q = rng.standard_normal((B, H, D)).astype(np.float32)
    scale = 1 / np.sqrt(D)
    if kind == "wide":
        q *= 8
    elif kind in ("tiny", "huge"):
        q *= np.float32(2.0 ** (-124 if kind == "tiny" else 120))
        scale = 2.0 ** (120 if kind == "tiny" else -122)
    elif kind == "spread":
        q *= np.exp2(-40 * rng.random((B, H, D))).astype(np.float32)
    else:
        q[0, 1, 5], q[1, H - 1, 127] = np.inf, np.nan
    q_bits = round_to_storage(q, "bf16")
    d_q = torch.from_numpy(q_bits.view(np.int16)).view(torch.bfloat16).to(DEV)
    out, lse = torch.zeros((B, H, D), device=DEV), torch.zeros((B, H), device=DEV)
    desc = ssa.make_desc(d_q, p.k, p.v, out, scale=scale)
    ws = torch.empty(ssa.decode_workspace_bytes(desc, T), dtype=torch.uint8, device=DEV)
    ctx = [T, 4321]
    ssa.decode_attn_dense(desc, d_q, p.k, p.v, torch.tensor(ctx, dtype=torch.int32, device=DEV), out, lse, ws)
    torch.cuda.synchronize()
    got, got_lse = out.double().cpu().numpy(), lse.double().cpu().numpy()
    bad = ~np.isfinite(q).all(axis=-1)
    assert np.isnan(got[bad]).all() and np.isnan(got_lse[bad]).all()
    q_bits[bad] = 0
    ref, ref_lse = O.decode_attn_dense(q_bits, *p.oracle_kv(), ctx, scale, "bf16/e4m3")
    assert float(np.linalg.norm((got - ref)[~bad])) <= 4e-6 * float(np.linalg.norm(ref[~bad]))
    np.testing.assert_allclose(got_lse[~bad], ref_lse[~bad], rtol=2e-6, atol=2e-6)


@pytest.mark.parametrize("group,T,top", [
    (2, 8000, 31), (8, 8000, 60), (12, 8000, 36), (20, 8000, 31), (33, 8000, 60), (8, 76000, 36), (20, 38000, 36)])
def test_shared_rows_over_an_8_bit_cache_with_keys_of_zero_where_the_query_is_largest(group, T, top):
    """A head dimension that K does not use (zeros: a narrower head padded to 128) leaves q free there: its size must not
    cost the other dimensions anything.  Every third query row has elements near 2^top there and a zero weight in every score;
    the others are ordinary.  The products left are those of ordinary rows, so the bound is theirs: scores of N(0, 1) carry
    2^-24 sqrt(128) relative, the rows at most four times that, 3e-6 in the 2-norm."""
    B, Hkv, D = 2, 2, 128
    H = group * Hkv
    p = Fp8Problem(B, H, Hkv, T, D, seed=group + top)
    rng = np.random.default_rng(top)
    p.k_bits[..., 96:] = 0
    p.k = torch.from_numpy(p.k_bits).view(torch.float8_e4m3fn).to(DEV)
    q = rng.standard_normal((B, H, D)).astype(np.float32)
    q[:, ::3, 96:] *= np.float32(2.0 ** top)
    q_bits = round_to_storage(q, "bf16")
    d_q = torch.from_numpy(q_bits.view(np.int16)).view(torch.bfloat16).to(DEV)
    out, lse = torch.zeros((B, H, D), device=DEV), torch.zeros((B, H), device=DEV)
    desc = ssa.make_desc(d_q, p.k, p.v, out)
    ws = torch.empty(max(ssa.decode_workspace_bytes(desc, T), ssa.decode_spans_workspace_bytes(desc, T, 2)),
                     dtype=torch.uint8, device=DEV)
    ctx = [T, 4321]
    d_ctx = torch.tensor(ctx, dtype=torch.int32, device=DEV)
    ref, ref_lse = O.decode_attn_dense(q_bits, *p.oracle_kv(), ctx, 1 / np.sqrt(D), "bf16/e4m3")
    index = torch.arange(T, dtype=torch.int32, device=DEV).expand(B, T).contiguous()
    spans = torch.tensor([[0, 100], [100, T]] * B, dtype=torch.int32, device=DEV)
    offs = torch.tensor([0, 2, 4], dtype=torch.int32, device=DEV)
    for call in (lambda: ssa.decode_attn_dense(desc, d_q, p.k, p.v, d_ctx, out, lse, ws),
                 lambda: ssa.decode_attn_sparse(desc, d_q, p.k, p.v, d_ctx, index, d_ctx, T, out, lse, ws),
                 lambda: ssa.decode_attn_spans(desc, d_q, p.k, p.v, d_ctx, offs, spans, 2, T, out, lse, None, None, ws)):
        call()
        torch.cuda.synchronize()
        assert float(np.linalg.norm(out.double().cpu().numpy() - ref)) <= 3e-6 * float(np.linalg.norm(ref))
        np.testing.assert_allclose(lse.double().cpu().numpy(), ref_lse, rtol=2e-6, atol=2e-6)
        out.zero_()
