"""What blocks do before the launch in front of theirs has ended: they prefetch by lists, lengths and page tables that may still be
a former step's, or no list at all.  Whatever these say, results are those of the lists as the launch in front leaves them."""
import numpy as np
import pytest
import torch

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
def test_lists_that_the_launch_in_front_still_writes(B, H, Hkv, D, rows, page_size, before):
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
    for sp, out in zip(spans, outs):                     # every launch's lists are written by the one in front
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
