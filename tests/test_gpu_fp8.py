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
    (3, 2, 140, [1, 16, 129]),          # list ends around a 16-row tile and around a round of the block's tiles
    (2, 7, 1100, [1023, 1025]),         # ... and around the staging window; a head tile with one head missing
    (3, 8, 700, [15, 17, 700]),
    (3, 9, 700, [127, 128, 0]),         # two head tiles, the second with one head; an empty list
    (2, 16, 2600, [2600, 513]),
    (3, 2, 51000, [51000, 1, 20000]),   # even shares of the full context
    (40, 4, 300, None),                 # one unit for most SMs: the large blocks, index and span lists
])
def test_grouped_heads_over_an_8_bit_cache(B, group, T, counts):
    # fp32 output: weights carry 22 bits or an absolute 2^-37, sums are fp32 over at most 51000 rows: 2^-22 per weight
    # and 2^-24 sqrt(51000) = 1.4e-5 relative per sum bound the error of an N(0, 1) average by 1.5e-5; 2e-5 is asserted
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
    ws = torch.empty(ssa.decode_spans_workspace_bytes(desc, T, 4), dtype=torch.uint8, device=DEV)
    ko, vo = p.oracle_kv()

    def check(ref, ref_lse, what):
        torch.cuda.synchronize()
        assert float(np.abs(out.double().cpu().numpy() - ref).max()) <= 2e-5, what
        ok = np.isfinite(ref_lse)
        np.testing.assert_allclose(lse.double().cpu().numpy()[ok], ref_lse[ok], rtol=2e-6, atol=2e-6, err_msg=what)
        assert int(status.item()) == 0

    ssa.decode_attn_sparse(desc, p.q, p.k, p.v, d_ctx, torch.from_numpy(index).to(DEV),
                           torch.tensor(counts, dtype=torch.int32, device=DEV), T, out, lse, ws, status)
    check(*O.decode_attn_sparse(p.q_bits, ko, vo, ctx, index, counts, 1 / np.sqrt(D), "bf16/e4m3"), "index lists")
    ssa.decode_attn_dense(desc, p.q, p.k, p.v, d_ctx, out, lse, ws, status)
    dense = O.decode_attn_dense(p.q_bits, ko, vo, ctx, 1 / np.sqrt(D), "bf16/e4m3")
    check(*dense, "full context")
    flat = torch.tensor([[0, T // 2], [T // 2, T]] * B, dtype=torch.int32, device=DEV)
    offs = torch.arange(0, 2 * B + 1, 2, dtype=torch.int32, device=DEV)
    ssa.decode_attn_spans(desc, p.q, p.k, p.v, d_ctx, offs, flat, 4, T, out, lse, None, None, ws, status)
    check(*dense, "span lists")


@pytest.mark.parametrize("group", [4, 12])
def test_grouped_heads_read_every_e4m3_pattern_exactly(group):
    """One selected row per K/V head: every head of the group returns that V row, exactly; a NaN in K or V shows."""
    B, Hkv, T, D = 1, 2, 32, 128
    H = group * Hkv
    p = Fp8Problem(B, H, Hkv, T, D, seed=3)
    pats = np.array([x for x in range(256) if x not in (0x7F, 0xFF)], np.uint8)
    v = p.v_bits.copy()
    v[0, 0, 5], v[0, 1, 5] = pats[:128], pats[126:254]
    out = torch.zeros((B, H, D), dtype=torch.float32, device=DEV)
    desc = ssa.make_desc(p.q, p.k, p.v, out)
    ws = torch.empty(ssa.decode_workspace_bytes(desc, 32), dtype=torch.uint8, device=DEV)
    idx = torch.full((1, 32), 5, dtype=torch.int32, device=DEV)
    one, ctx = (torch.tensor([x], dtype=torch.int32, device=DEV) for x in (1, T))

    def run(v_bits):
        pv = torch.from_numpy(v_bits).view(torch.float8_e4m3fn).to(DEV)
        ssa.decode_attn_sparse(desc, p.q, p.k, pv, ctx, idx, one, 32, out, None, ws, None)
        torch.cuda.synchronize()
        return out.double().cpu().numpy()[0]

    want = np.repeat(O.decode_e4m3(v[0, :, 5]), group, axis=0)
    assert np.array_equal(run(v), want)
    v[0, 0, 5, 77] = 0x7F
    got = run(v)
    assert np.isnan(got[:group, 77]).all() and np.isfinite(np.delete(got, 77, axis=1)).all()
