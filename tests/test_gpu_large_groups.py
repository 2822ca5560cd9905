"""More than sixteen query heads (or head, token pairs) per K/V head: several row-sharing blocks per chunk, or one head per
block where a launch is small, against the fp64 oracle."""
import numpy as np
import pytest
import torch

from oracle import ssa_oracle as O
from paper_2404_09336_b200 import ssa
from paper_2404_09336_b200.runner import bits_to_tensor

from gpu_util import DEV, random_bits
from test_gpu_fp8 import Fp8Problem

pytestmark = pytest.mark.gpu


def problem(dtype, B, H, Hkv, T, seed):
    if dtype == "fp8":
        p = Fp8Problem(B, H, Hkv, T, 128, seed)
        return p.q, p.k, p.v, p.q_bits, p.k_bits, p.v_bits, "bf16/e4m3"
    rng = np.random.default_rng(seed)
    bits = [random_bits(rng, s, dtype) for s in ((B, H, 128), (B, Hkv, T, 128), (B, Hkv, T, 128))]
    return (*(bits_to_tensor(x, dtype).to(DEV) for x in bits), *bits, dtype)


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
    """fp32 output.  Weights carry 22 bits or more (or an absolute 2^-37), a tile's products are summed on their own, sums
    are fp32: independent errors of 2^-22 per weight or product stay below 2.4e-7 of the result in the 2-norm (measured:
    1.0e-7..1.9e-7; one head per block 1.4e-7..2.5e-7); four times that is asserted."""
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
    """A workspace sized by another bound, too small for the row-sharing plan, is taken as before; so is the call without one."""
    B, H, Hkv, T, D = 1, 120, 6, 2000, 128
    q, k, v, qb, kb, vb, name = problem("bf16", B, H, Hkv, T, seed=1)
    out = torch.zeros((B, H, D), dtype=torch.float32, device=DEV)
    desc = ssa.make_desc(q, k, v, out)
    idx = torch.arange(T, dtype=torch.int32, device=DEV).view(1, T)
    d_ctx, d_cnt = (torch.tensor([T], dtype=torch.int32, device=DEV) for _ in range(2))
    ref, _ = O.decode_attn_dense(qb, np.repeat(kb, 20, axis=1), np.repeat(vb, 20, axis=1), [T], 1 / np.sqrt(D), name)

    def check():
        torch.cuda.synchronize()
        assert float(np.linalg.norm(out.double().cpu().numpy() - ref)) <= 1e-6 * float(np.linalg.norm(ref))
        out.zero_()

    for nbytes in (ssa.decode_workspace_bytes(desc, T), sum((H * 8 * n + 255) // 256 * 256 for n in (4 * D, 8))):
        ws = torch.full((nbytes + 4096,), 0xA5, dtype=torch.uint8, device=DEV)
        ssa.decode_attn_sparse(desc, q, k, v, d_ctx, idx, d_cnt, T, out, None, ws[:nbytes], None)
        check()
        assert bool((ws[nbytes:] == 0xA5).all())
    ssa.decode_attn_sparse_noalloc(desc, q, k, v, d_ctx, idx, d_cnt, T, out, None, None)
    check()
