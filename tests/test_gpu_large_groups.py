"""More than sixteen query heads (or head, token pairs) per K/V head: several row-sharing blocks per chunk, or one head per
block where a launch is small, against the fp64 oracle."""
import numpy as np
import pytest
import torch

from oracle import ssa_oracle as O
from paper_2404_09336_b200 import ssa
from paper_2404_09336_b200.inputs import round_to_storage
from paper_2404_09336_b200.runner import bits_to_tensor

from gpu_util import DEV, random_bits
from test_gpu_fp8 import Fp8Problem, to_e4m3_bits

pytestmark = pytest.mark.gpu


def problem(dtype, B, H, Hkv, T, seed):
    if dtype == "fp8":
        p = Fp8Problem(B, H, Hkv, T, 128, seed)
        return p.q, p.k, p.v, p.q_bits, p.k_bits, p.v_bits, "bf16/e4m3"
    rng = np.random.default_rng(seed)
    bits = [random_bits(rng, s, dtype) for s in ((B, H, 128), (B, Hkv, T, 128), (B, Hkv, T, 128))]
    return (*(bits_to_tensor(x, dtype).to(DEV) for x in bits), *bits, dtype)


def upload(dtype, q_bits, k_bits, v_bits):
    if dtype != "fp8":
        return tuple(bits_to_tensor(x, dtype).to(DEV) for x in (q_bits, k_bits, v_bits))
    return (bits_to_tensor(q_bits, "bf16").to(DEV),
            *(torch.from_numpy(x).view(torch.float8_e4m3fn).to(DEV) for x in (k_bits, v_bits)))


@pytest.mark.parametrize("dtype,B,Hkv,G,T,counts", [
    ("bf16", 1, 1, 17, 300, [129]),                             # small: one head per block
    ("bf16", 3, 3, 17, 1300, [1300, 0, 17]),                    # 9 + 8 heads, several chunks; an empty list
    ("f16", 2, 4, 24, 1100, [1023, 16]),                        # 12 + 12
    ("fp8", 2, 2, 33, 2500, [2500, 513]),                       # 3 x 11
    ("bf16", 30, 2, 32, 300, None),                             # one large block per SM
    ("f16", 150, 1, 20, 70, None),                              # a block per request and part, no second pass
    ("f16", 2, 1, 40, 52000, [5, 40000]), ("bf16", 1, 2, 17, 76000, [76000]),   # full contexts cut on the device
    ("fp8", 2, 2, 32, 38000, [129, 1000]),
])
def test_large_groups_against_the_oracle(dtype, B, Hkv, G, T, counts):
    """fp32 output.  Weights carry 23 bits or more, a tile's products are summed on their own, sums are fp32: independent errors
    of 2^-22 per weight or product stay below 2.4e-7 of the result in the 2-norm (measured: 1.0e-7..1.9e-7; one head per block
    1.4e-7..2.5e-7); four times that is asserted."""
    H, D = G * Hkv, 128
    q, k, v, qb, kb, vb, name = problem(dtype, B, H, Hkv, T, seed=G + T)
    rng = np.random.default_rng(T)
    counts = counts or [int(x) for x in rng.integers(1, T + 1, size=B)]
    index = np.full((B, T), -1, np.int32)
    for b, c in enumerate(counts):
        index[b, :c] = np.sort(rng.choice(T, c, replace=False))
    out = torch.full((B, H, D), 7.0, dtype=torch.float32, device=DEV)
    lse = torch.full((B, H), 7.0, dtype=torch.float32, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    desc = ssa.make_desc(q, k, v, out)
    need = max(ssa.decode_spans_workspace_bytes(desc, T, 4), ssa.decode_workspace_bytes(desc, T))
    ws = torch.full((need + 4096,), 0xA5, dtype=torch.uint8, device=DEV)
    d_ctx, d_cnt = (torch.tensor(x, dtype=torch.int32, device=DEV) for x in ([T] * B, counts))
    d_idx = torch.from_numpy(index).to(DEV)
    scale = 1 / np.sqrt(D)
    seqs = sorted({0, 1, B // 2, B - 1} & set(range(B)))

    def check(ref, ref_lse, what):
        torch.cuda.synchronize()
        diff = (out.double().cpu().numpy() - ref)[seqs]
        assert float(np.linalg.norm(diff)) <= 1e-6 * float(np.linalg.norm(ref[seqs])), what
        ok = np.isfinite(ref_lse[seqs])
        got = lse.double().cpu().numpy()[seqs]
        np.testing.assert_allclose(got[ok], ref_lse[seqs][ok], rtol=2e-6, atol=2e-6, err_msg=what)
        assert np.all(np.isneginf(got[~ok])), what
        assert int(status.item()) == 0 and bool((ws[need:] == 0xA5).all())
        out.fill_(7.0)

    ko, vo = np.repeat(kb, G, axis=1), np.repeat(vb, G, axis=1)
    listed = O.decode_attn_sparse(qb, ko, vo, [T] * B, index, counts, scale, name, seqs=seqs)
    ssa.decode_attn_sparse(desc, q, k, v, d_ctx, d_idx, d_cnt, T, out, lse, ws[:need], status)
    check(*listed, "index lists")
    pages = [x.transpose(1, 2).reshape(B * T, 1, Hkv, D).contiguous() for x in (k.view(torch.uint8), v.view(torch.uint8))] \
        if dtype == "fp8" else [x.transpose(1, 2).reshape(B * T, 1, Hkv, D).contiguous() for x in (k, v)]
    kp, vp = (x.view(k.dtype) for x in pages)
    table = torch.arange(B * T, dtype=torch.int32, device=DEV).view(B, T)
    paging = ssa.make_paging(table, 1, B * T)
    ssa.decode_attn_sparse_paged(ssa.make_desc_paged(q, kp, vp, out, T), q, kp, vp, paging, d_ctx, d_idx, d_cnt, T, out, lse,
                                 ws[:need], status)
    check(*listed, "a paged cache")
    ragged = [min(T, T // 64 + 64 * (b % 3)) if b else T for b in range(B)]
    ssa.decode_attn_dense(desc, q, k, v, torch.tensor(ragged, dtype=torch.int32, device=DEV), out, lse, ws[:need], status)
    check(*O.decode_attn_dense(qb, ko, vo, ragged, scale, name, seqs=seqs), "full contexts")
    flat = torch.tensor([[0, T // 2], [T // 2, T]] * B, dtype=torch.int32, device=DEV)
    offs = torch.arange(0, 2 * B + 1, 2, dtype=torch.int32, device=DEV)
    d_index, d_counts = torch.full((B, T), -7, dtype=torch.int32, device=DEV), torch.zeros(B, dtype=torch.int32, device=DEV)
    ssa.decode_attn_spans(desc, q, k, v, d_ctx, offs, flat, 4, T, out, lse, d_index, d_counts, ws[:need], status)
    check(*O.decode_attn_dense(qb, ko, vo, [T] * B, scale, name, seqs=seqs), "span lists")
    assert d_counts.tolist() == [T] * B and torch.equal(d_index.cpu(), torch.arange(T, dtype=torch.int32).expand(B, T))


def test_large_group_in_the_workspace_of_one_head_per_block():
    """A workspace sized by another bound, too small for the row-sharing plan, is taken as before: lists of 1000 rows are then
    one chunk per head, 200 partial results, instead of four chunks and a second pass.  The call without a workspace goes by
    the one-head plan as well: it refuses what that does not fit, though the row-sharing one would."""
    B, H, Hkv, T, D = 1, 200, 10, 1000, 128
    q, k, v, qb, kb, vb, name = problem("bf16", B, H, Hkv, T, seed=1)
    out = torch.zeros((B, H, D), dtype=torch.float32, device=DEV)
    desc = ssa.make_desc(q, k, v, out)
    idx = torch.arange(T, dtype=torch.int32, device=DEV).view(1, T)
    d_ctx, d_cnt = (torch.tensor([T], dtype=torch.int32, device=DEV) for _ in range(2))
    ref, _ = O.decode_attn_dense(qb, np.repeat(kb, 20, axis=1), np.repeat(vb, 20, axis=1), [T], 1 / np.sqrt(D), name)
    full, small = ssa.decode_workspace_bytes(desc, T), sum((H * 4 * n + 255) // 256 * 256 for n in (D, 2))
    assert small < H * 4 * (4 * D + 8) <= full                    # four chunks per head do not fit

    def check(before, launches):
        assert ssa.launch_count() - before == launches
        torch.cuda.synchronize()
        assert float(np.linalg.norm(out.double().cpu().numpy() - ref)) <= 1e-6 * float(np.linalg.norm(ref))
        out.zero_()

    ws = torch.empty(full + 4096, dtype=torch.uint8, device=DEV)
    for nbytes, launches in ((full, 2), (small, 1)):
        ws.fill_(0xA5)
        before = ssa.launch_count()
        ssa.decode_attn_sparse(desc, q, k, v, d_ctx, idx, d_cnt, T, out, None, ws[:nbytes], None)
        check(before, launches)
        assert bool((ws[nbytes:] == 0xA5).all())
    assert ssa.decode_attn_sparse(desc, q, k, v, d_ctx, idx, d_cnt, T, out, None, ws[:small - 256], None,
                                  check=False) == ssa.ERR_WORKSPACE
    # span lists, few of them and more than a block merges on chip (their index list then shares the workspace)
    for n, lists in ((2, 256), (T, 256 + 4 * 1024)):
        spans = torch.tensor([[T * i // n, T * (i + 1) // n] for i in range(n)], dtype=torch.int32, device=DEV)
        offs, nbytes = torch.tensor([0, n], dtype=torch.int32, device=DEV), small + lists
        ws.fill_(0xA5)
        before = ssa.launch_count()
        ssa.decode_attn_spans(desc, q, k, v, d_ctx, offs, spans, n, T, out, None, None, None, ws[:nbytes], None)
        check(before, 1 if n == 2 else 2)
        assert bool((ws[nbytes:] == 0xA5).all())
        assert ssa.decode_attn_spans(desc, q, k, v, d_ctx, offs, spans, n, T, out, None, None, None, ws[:nbytes - 256], None,
                                     check=False) == ssa.ERR_WORKSPACE
    before = ssa.launch_count()
    ssa.decode_attn_sparse_noalloc(desc, q, k, v, d_ctx, idx, d_cnt, T, out, None, None)
    check(before, 2)
    desc.B, desc.max_ctx = 2, 16000                                # 400 heads x 63 chunks of 256 rows
    assert ssa.decode_attn_sparse_noalloc(desc, q, k, v, d_ctx, torch.zeros((2, 16000), dtype=torch.int32, device=DEV), d_cnt,
                                          16000, out, None, None, check=False) == ssa.ERR_WORKSPACE


# dtype, B, Hkv, G, T: lists (one large block per SM, several chunks, one block) and full contexts, those of the last two cut
# on the device
SHAPES = [("bf16", 30, 2, 32, 300), ("f16", 2, 4, 24, 1100), ("fp8", 2, 2, 33, 2500), ("f16", 150, 1, 20, 70),
          ("f16", 1, 1, 20, 76000), ("bf16", 1, 2, 17, 76000), ("fp8", 1, 2, 32, 38000)]


class _PerHead:
    """A cache of K/V heads, looked up by query head."""

    def __init__(self, bits, group):
        self.bits, self.group = bits, group

    def __getitem__(self, at):
        return self.bits[at[0], at[1] // self.group]


def reference(q_bits, k_bits, v_bits, B, T, G, scale, name):
    """Full contexts of the first, the middle and the last request, first and last heads of the first and the last K/V head."""
    H = q_bits.shape[1]
    kv = (_PerHead(x, G) for x in (k_bits, v_bits))
    with np.errstate(invalid="ignore"):                 # (infinities of both signs make a NaN)
        return O.decode_attn_dense(q_bits, *kv, [T] * B, scale, name, heads=sorted({0, G - 1, H - G, H - 1}),
                                   seqs=sorted({0, B // 2, B - 1}))


def all_calls(desc, q, k, v, T, out, lse):
    """Index lists, a paged cache, span lists (by every warp and by one) and full contexts of all T rows."""
    B, Hkv, D = q.shape[0], k.shape[1], q.shape[2]
    need = max(ssa.decode_spans_workspace_bytes(desc, T, 40), ssa.decode_workspace_bytes(desc, T))
    ws = torch.empty(need, dtype=torch.uint8, device=DEV)
    ctx = torch.full((B,), T, dtype=torch.int32, device=DEV)
    index = torch.arange(T, dtype=torch.int32, device=DEV).expand(B, T).contiguous()
    raw = (lambda x: x.view(torch.uint8)) if k.element_size() == 1 else (lambda x: x)
    kp, vp = (raw(x).transpose(1, 2).reshape(B * T, 1, Hkv, D).contiguous().view(x.dtype) for x in (k, v))
    table = torch.arange(B * T, dtype=torch.int32, device=DEV).view(B, T)
    paging, paged = ssa.make_paging(table, 1, B * T), ssa.make_desc_paged(q, kp, vp, out, T, scale=desc.scale)
    few = torch.tensor([[0, T // 2], [T // 2, T]] * B, dtype=torch.int32, device=DEV)
    many = torch.tensor([[0, T // 2]] * 38 + [[T // 2, T], [5, 9]], dtype=torch.int32, device=DEV).repeat(B, 1)
    step = lambda n: torch.arange(0, n * B + 1, n, dtype=torch.int32, device=DEV)
    yield "index lists", lambda: ssa.decode_attn_sparse(desc, q, k, v, ctx, index, ctx, T, out, lse, ws)
    yield "a paged cache", lambda: ssa.decode_attn_sparse_paged(paged, q, kp, vp, paging, ctx, index, ctx, T, out, lse, ws)
    yield "full contexts", lambda: ssa.decode_attn_dense(desc, q, k, v, ctx, out, lse, ws)
    yield "few spans", lambda: ssa.decode_attn_spans(desc, q, k, v, ctx, step(2), few, 2, T, out, lse, None, None, ws)
    yield "many spans", lambda: ssa.decode_attn_spans(desc, q, k, v, ctx, step(40), many, 40, T, out, lse, None, None, ws)


@pytest.mark.parametrize("dtype,B,Hkv,G,T", SHAPES)
def test_rows_far_below_the_largest_weight_of_a_large_group(dtype, B, Hkv, G, T):
    """Every seventh row has a score 20 above the others' (every 21st, 40) and a V row of zeros, so the output is what the
    light rows add: their weights, 2^-29 and 2^-58 of the largest, must be fp32 values like all others and not be cut off.
    Bound: scores of 40 are 58 in log2 units, where fp32 values lie 2^-18 apart: 2.7e-6 of a weight; 1e-5 is asserted."""
    H, D = G * Hkv, 128
    q, k, v, qb, kb, vb, name = problem(dtype, B, H, Hkv, T, seed=T)
    bits = lambda x, what: (to_e4m3_bits if what == "fp8" else lambda y: round_to_storage(y, what))(np.full(1, x, np.float32))[0]
    qb[..., 0], kb[..., 0] = bits(8, "bf16" if dtype == "fp8" else dtype), 0
    heavy = np.arange(0, T, 7)
    kb[:, :, heavy, 0], kb[:, :, heavy[::3], 0], vb[:, :, heavy] = bits(20, dtype), bits(40, dtype), 0
    q, k, v = upload(dtype, qb, kb, vb)
    out, lse = torch.zeros((B, H, D), device=DEV), torch.zeros((B, H), device=DEV)
    desc = ssa.make_desc(q, k, v, out, scale=0.125)
    ref, ref_lse = reference(qb, kb, vb, B, T, G, 0.125, name)
    some = ~np.isnan(ref_lse)
    assert 0 < np.abs(ref[some]).max() < 2.0 ** -50
    for what, call in all_calls(desc, q, k, v, T, out, lse):
        call()
        torch.cuda.synchronize()
        got = out.double().cpu().numpy()[some]
        assert float(np.linalg.norm(got - ref[some])) <= 1e-5 * float(np.linalg.norm(ref[some])), what
        np.testing.assert_allclose(lse.double().cpu().numpy()[some], ref_lse[some], rtol=2e-6, atol=2e-6, err_msg=what)
        out.fill_(7.0)


@pytest.mark.parametrize("dtype,B,Hkv,G,T", [s for s in SHAPES if s[0] != "fp8"])
def test_infinities_in_v_reach_the_rows_of_a_large_group(dtype, B, Hkv, G, T):
    """An infinity in a selected row of V is one in the output, two of different sign or a NaN make a NaN, and no other dim is
    touched; a NaN in K makes the rows of its heads NaN.  As one head per block has it."""
    H, D = G * Hkv, 128
    q, k, v, qb, kb, vb, name = problem(dtype, B, H, Hkv, T, seed=T + 1)
    inf, nan = ({"bf16": 0x7F80, "f16": 0x7C00}[dtype], {"bf16": 0x7FC0, "f16": 0x7E00}[dtype])
    vb[:, 0, T // 3, 5], vb[:, 0, T - 1, 6], vb[:, 0, 0, 6] = inf, inf | 0x8000, inf | 0x8000
    vb[:, 0, 1, 7], vb[:, 0, T - 2, 7], vb[:, 0, T // 2, 126] = inf, inf | 0x8000, nan
    vb[:, Hkv - 1, T // 2 + 1, 127] = inf
    q, k, v = upload(dtype, qb, kb, vb)
    out, lse = torch.zeros((B, H, D), device=DEV), torch.zeros((B, H), device=DEV)
    desc = ssa.make_desc(q, k, v, out)
    ref, ref_lse = reference(qb, kb, vb, B, T, G, 1 / np.sqrt(D), name)
    some = ~np.isnan(ref_lse)
    some_first, some_last = some & (np.arange(H) < G), some & (np.arange(H) >= H - G)
    assert np.isposinf(ref[some_first][:, 5]).all() and np.isneginf(ref[some_first][:, 6]).all()
    assert np.isnan(ref[some_first][:, [7, 126]]).all() and np.isposinf(ref[some_last][:, 127]).all()
    for what, call in all_calls(desc, q, k, v, T, out, lse):
        call()
        torch.cuda.synchronize()
        np.testing.assert_allclose(out.double().cpu().numpy()[some], ref[some], rtol=1e-4, atol=1e-5, err_msg=what)
        np.testing.assert_allclose(lse.double().cpu().numpy()[some], ref_lse[some], rtol=2e-6, atol=2e-6, err_msg=what)
        out.fill_(7.0)
    kb[:, 0, T // 4, 9] = nan
    q, k, v = upload(dtype, qb, kb, vb)
    for what, call in all_calls(desc, q, k, v, T, out, lse):
        call()
        torch.cuda.synchronize()
        assert bool(out[:, :G].isnan().all()) and bool(lse[:, :G].isnan().all()), what
        if Hkv > 1:
            got = out.double().cpu().numpy()[some_last]
            np.testing.assert_allclose(got, ref[some_last], rtol=1e-4, atol=1e-5, err_msg=what)
