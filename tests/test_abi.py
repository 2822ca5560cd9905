"""The C-ABI library loads, exports what include/ssa.h declares, and rejects
bad arguments on the host before anything is launched (no GPU needed)."""
import ctypes as C
import os
import re
import shutil
import subprocess

import pytest
import torch

from paper_2404_09336_b200 import build, ssa

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def declared_symbols():
    text = open(os.path.join(ROOT, "include", "ssa.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(ssa_[a-z0-9_]+)\s*\(", text)))


def test_every_declared_symbol_is_exported():
    names = declared_symbols()
    assert {"ssa_spans_to_index", "ssa_decode_attn_sparse", "ssa_decode_attn_dense",
            "ssa_decode_workspace_bytes"} <= set(names)
    raw = C.CDLL(ssa.LIBRARY_PATH)
    for n in names:
        assert hasattr(raw, n), n


def test_library_is_in_tree():
    assert os.path.dirname(ssa.LIBRARY_PATH) == os.path.join(ROOT, "paper_2404_09336_b200")


def test_version_and_strings():
    assert ssa.version() >= 100
    assert ssa.status_string(ssa.OK) == "ok"
    assert "aligned" in ssa.status_string(ssa.ERR_ALIGN)
    assert "unknown" in ssa.status_string(12345)


def good_desc():
    d = ssa.AttnDesc()
    d.B, d.H, d.H_kv, d.D, d.max_ctx = 2, 4, 4, 128, 512
    d.kv_dtype, d.out_dtype, d.scale = ssa.BF16, ssa.BF16, 0.0
    d.q_stride_b, d.q_stride_h = 4 * 128, 128
    d.k_stride_b, d.k_stride_h, d.k_stride_t = 4 * 512 * 128, 512 * 128, 128
    d.v_stride_b, d.v_stride_h, d.v_stride_t = 4 * 512 * 128, 512 * 128, 128
    d.o_stride_b, d.o_stride_h = 4 * 128, 128
    return d


def test_workspace_query():
    d = good_desc()
    small = ssa.decode_workspace_bytes(d, 64)
    full = ssa.decode_workspace_bytes(d, 512)
    assert 0 < small <= full
    assert full >= 2 * 4 * (512 // 256) * (128 * 4 + 8)
    d.D = 96
    assert ssa.decode_workspace_bytes(d, 64) == 0
    d = good_desc()
    assert ssa.decode_workspace_bytes(d, 0) == 0


def test_small_grouped_launches_over_an_8_bit_cache_are_planned_one_head_per_block():
    """Partial results (one row of D floats and a pair per chunk and head) show the plan: 820 rows, 32 query heads over 2
    cache heads are 13 chunks per head, shared rows would be 4; over 8 cache heads sharing pays already; a 16-bit cache
    always shares."""
    def triples(H_kv, kv_dtype, sel=820):
        d = good_desc()
        d.B, d.H, d.H_kv, d.max_ctx, d.kv_dtype, d.out_dtype = 1, 32, H_kv, 8192, kv_dtype, ssa.F32
        return ssa.decode_workspace_bytes(d, sel) // (4 * 128 + 8)

    assert triples(2, ssa.FP8_E4M3) == 32 * 13
    assert triples(8, ssa.FP8_E4M3) == 32 * 4
    assert triples(2, ssa.BF16) == triples(8, ssa.BF16) == 32 * 4
    assert triples(2, ssa.FP8_E4M3, 40) == triples(2, ssa.BF16, 40) == 32


P = C.c_void_p(0x1000)      # never dereferenced: validation fails first
NUL = None


def sparse(d, q=P, k=P, v=P, ctx=P, idx=P, stride=64, cnt=P, max_sel=64, out=P, ws=P, ws_bytes=1 << 30):
    return ssa.lib.ssa_decode_attn_sparse(C.byref(d), q, k, v, ctx, idx, stride, cnt, max_sel, out, NUL, ws,
                                          ws_bytes, NUL, NUL)


def test_sparse_rejects_bad_arguments_without_launching():
    before = ssa.launch_count()
    d = good_desc()
    assert ssa.lib.ssa_decode_attn_sparse(None, P, P, P, P, P, 64, P, 64, P, NUL, P, 1 << 30, NUL, NUL) == ssa.ERR_NULL
    assert sparse(d, q=NUL) == ssa.ERR_NULL
    assert sparse(d, idx=NUL) == ssa.ERR_NULL
    assert sparse(d, out=NUL) == ssa.ERR_NULL
    assert sparse(d, max_sel=65) == ssa.ERR_CAPACITY
    assert sparse(d, max_sel=0) == ssa.ERR_CAPACITY
    assert sparse(d, stride=0) == ssa.ERR_CAPACITY
    assert sparse(d, k=C.c_void_p(0x1008)) == ssa.ERR_ALIGN
    assert sparse(d, ws=NUL) == ssa.ERR_WORKSPACE
    assert sparse(d, ws_bytes=16) == ssa.ERR_WORKSPACE
    for field, val, err in [("D", 96, ssa.ERR_UNSUPPORTED), ("H_kv", 3, ssa.ERR_UNSUPPORTED),
                            ("kv_dtype", ssa.F32, ssa.ERR_DTYPE), ("out_dtype", ssa.F16, ssa.ERR_DTYPE),
                            ("k_stride_t", 132, ssa.ERR_ALIGN), ("B", 0, ssa.ERR_SHAPE),
                            ("max_ctx", 0, ssa.ERR_SHAPE), ("v_stride_h", -128, ssa.ERR_SHAPE)]:
        d = good_desc()
        setattr(d, field, val)
        assert sparse(d) == err, field
    assert ssa.launch_count() == before


def test_dense_and_index_reject_bad_arguments():
    before = ssa.launch_count()
    d = good_desc()
    f = ssa.lib.ssa_decode_attn_dense
    assert f(C.byref(d), P, P, P, NUL, P, NUL, P, 1 << 30, NUL, NUL) == ssa.ERR_NULL
    assert f(C.byref(d), P, P, P, P, P, NUL, P, 64, NUL, NUL) == ssa.ERR_WORKSPACE
    d.D = 32
    assert f(C.byref(d), P, P, P, P, P, NUL, P, 1 << 30, NUL, NUL) == ssa.ERR_UNSUPPORTED
    g = ssa.lib.ssa_spans_to_index
    assert g(NUL, P, P, 4, P, 64, P, NUL, NUL) == ssa.ERR_NULL
    assert g(P, P, P, 0, P, 64, P, NUL, NUL) == ssa.ERR_SHAPE
    assert g(P, P, P, 4, P, 0, P, NUL, NUL) == ssa.ERR_SHAPE
    assert g(P, C.c_void_p(0x1004), P, 4, P, 64, P, NUL, NUL) == ssa.ERR_ALIGN
    assert ssa.launch_count() == before


def test_error_raises_through_binding():
    with pytest.raises(ssa.SsaError) as e:
        ssa._check("ssa_decode_attn_sparse", ssa.ERR_WORKSPACE, True)
    assert "workspace" in str(e.value)


def test_step_rejects_bad_copy_requests_before_enqueuing_anything():
    d = good_desc()
    st = ssa.Step()
    assert ssa.lib.ssa_decode_step(None, C.byref(st), None) == ssa.ERR_NULL
    st.host_in, st.dev_in, st.in_bytes = 0x1000, None, 256
    assert ssa.decode_step(d, st, stream=0, check=False) == ssa.ERR_NULL         # a copy without a destination
    st.dev_in = 0x2000
    st.flags = 8
    assert ssa.decode_step(d, st, stream=0, check=False) == ssa.ERR_UNSUPPORTED  # unknown flag bit
    st.flags = ssa.STEP_ONE_KERNEL | ssa.STEP_TWO_KERNELS
    assert ssa.decode_step(d, st, stream=0, check=False) == ssa.ERR_UNSUPPORTED  # contradictory
    st.flags = ssa.STEP_COPY_BY_KERNEL
    st.host_in = 0x1008
    assert ssa.decode_step(d, st, stream=0, check=False) == ssa.ERR_ALIGN
    st.host_in, st.in_bytes = 0x1000, 250
    assert ssa.decode_step(d, st, stream=0, check=False) == ssa.ERR_ALIGN
    import numpy as np
    buf = np.zeros(4096 + 64, np.uint8)                                          # ordinary pageable memory
    addr = (buf.ctypes.data + 63) // 64 * 64
    st.host_in, st.in_bytes = addr, 256
    assert ssa.decode_step(d, st, stream=0, check=False) == ssa.ERR_UNSUPPORTED  # kernels cannot address it


def test_refs_to_index_rejects_bad_arguments():
    t = ssa.AnchorTables()
    for name, _ in t._fields_:
        setattr(t, name, 0x1000)
    call = lambda tab, B, index, stride, counts: ssa.lib.ssa_refs_to_index(
        C.byref(tab) if tab is not None else None, B, index, stride, counts, None, None)
    assert call(None, 1, 0x2000, 64, 0x3000) == ssa.ERR_NULL
    assert call(t, 1, None, 64, 0x3000) == ssa.ERR_NULL
    assert call(t, 0, 0x2000, 64, 0x3000) == ssa.ERR_SHAPE
    assert call(t, 70000, 0x2000, 64, 0x3000) == ssa.ERR_SHAPE
    assert call(t, 1, 0x2000, 0, 0x3000) == ssa.ERR_SHAPE
    t.refs = 0x1004
    assert call(t, 1, 0x2000, 64, 0x3000) == ssa.ERR_ALIGN
    t.refs, t.lines = 0x1000, None
    assert call(t, 1, 0x2000, 64, 0x3000) == ssa.ERR_NULL


def test_header_is_plain_c_and_cpp(tmp_path):
    # the boundary is a C ABI: the header must compile as C99 and as C++ with nothing but the standard headers
    import shutil
    import subprocess
    src = tmp_path / "use_ssa.c"
    src.write_text('#include "ssa.h"\n'
                   "int main(void) {\n"
                   "  ssa_attn_desc d; ssa_step s; ssa_anchor_tables t; ssa_paging p;\n"
                   "  (void)d; (void)s; (void)t; (void)p;\n"
                   "  return (int)(sizeof(ssa_step) == 0) + (SSA_MAX_SPANS_PER_SEQ != 2048);\n"
                   "}\n")
    inc = os.path.join(ROOT, "include")
    for cc, std in (("gcc", "-std=c99"), ("g++", "-std=c++11")):
        exe = shutil.which(cc)
        if exe is None:
            pytest.skip(f"{cc} not installed")
        args = [exe, std, "-Wall", "-Werror", "-pedantic", "-I", inc, "-fsyntax-only"]
        args += ["-x", "c++"] if cc == "g++" else []
        res = subprocess.run(args + [str(src)], capture_output=True, text=True)
        assert res.returncode == 0, res.stderr


def test_struct_layouts_of_the_binding_match_the_header(tmp_path):
    # sizes and a few offsets of the ctypes mirrors against what the C compiler lays out
    import shutil
    import subprocess
    if shutil.which("gcc") is None:
        pytest.skip("gcc not installed")
    src = tmp_path / "layout.c"
    src.write_text('#include <stdio.h>\n#include <stddef.h>\n#include "ssa.h"\n'
                   "int main(void) {\n"
                   '  printf("%zu %zu %zu %zu %zu %zu %zu %zu\\n", sizeof(ssa_attn_desc), sizeof(ssa_step),\n'
                   "         sizeof(ssa_anchor_tables), sizeof(ssa_paging), offsetof(ssa_attn_desc, scale),\n"
                   "         offsetof(ssa_step, flags), offsetof(ssa_step, host_in), offsetof(ssa_paging, n_pages));\n"
                   "  return 0;\n}\n")
    exe = tmp_path / "layout"
    subprocess.run(["gcc", "-I", os.path.join(ROOT, "include"), "-o", str(exe), str(src)], check=True)
    got = [int(x) for x in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()]
    want = [C.sizeof(ssa.AttnDesc), C.sizeof(ssa.Step), C.sizeof(ssa.AnchorTables), C.sizeof(ssa.Paging),
            ssa.AttnDesc.scale.offset, ssa.Step.flags.offset, ssa.Step.host_in.offset, ssa.Paging.n_pages.offset]
    assert got == want


def test_workspace_of_a_larger_batch_serves_smaller_ones():
    """A size asked for once, for the largest batch and the longest lists, holds what any smaller call needs: its partial
    results (a row of D floats and a pair per head and chunk) with one head per block, where that is the only plan and the
    size is the need; with shared rows, two blocks per SM at most, of 256 rows or more (148 SMs, also where there is none)."""
    rows = [1, 64, 65, 128, 200, 256, 257, 300, 400, 512, 513, 700, 768, 820, 1000, 1024, 1025, 1500, 2048, 2049, 4000, 16000]
    batches = [1, 2, 3, 4, 5, 6, 7, 9, 10, 12, 14, 16, 18, 20, 24, 28, 32, 37, 40, 48, 64, 148, 149, 200, 296, 297]
    up = lambda n, to: -(-n // to) * to

    def needed(d, r):
        G = d.H // d.H_kv
        if G == 1 or d.D == 64:
            return ssa.decode_workspace_bytes(d, r)
        units, n = d.B * d.H_kv * -(-G // 16), 1
        if not (148 < 2 * units and units <= 148 and r <= 2048):
            n = max(1, min(296 // units, -(-r // 256)))
            n = -(-r // up(-(-r // n), 64))
        return up(d.B * d.H * n * 4 * d.D, 256) + up(d.B * d.H * n * 8, 256)

    # (groups of 2 to 16 are older and go by their own need)
    for H, H_kv in ((8, 8), (32, 32), (10, 10), (1, 1), (136, 8), (96, 4), (24, 1), (17, 1), (200, 10)):
        for D in (64, 128):
            for kv in (ssa.F16, ssa.FP8_E4M3):
                most = [0] * len(rows)                  # needed by the batches so far, with up to rows[i] rows
                for B in batches:
                    for i, r in enumerate(rows):
                        d = good_desc()
                        d.B, d.H, d.H_kv, d.D, d.max_ctx, d.kv_dtype, d.out_dtype = B, H, H_kv, D, 20000, kv, ssa.F32
                        most[i] = max(most[i], most[max(i - 1, 0)], needed(d, r))
                        assert ssa.decode_workspace_bytes(d, r) >= most[i], (H, H_kv, D, kv, B, r)


@pytest.mark.skipif(torch.cuda.is_available() or shutil.which("nvcc") is None, reason="enters launches with addresses that are none")
@pytest.mark.parametrize("defines", [["-DSSA_MIN_BLOCKS=2"], ["-DSSA_WARPS=8", "-DSSA_MIN_BLOCKS=2"]])
def test_lists_are_taken_whole_only_by_blocks_that_can_stage_them(tmp_path, defines):
    """Blocks of the smallest size stage 512 entries.  With other block sizes (a build define) a launch of 200 heads may get no
    larger ones, and then 1000 rows must be cut.  The workspace of one partial result per head shows which: too small, or
    enough, so that the call goes on to a launch that this machine, without a GPU, refuses."""
    out = str(tmp_path / "libssa.so")
    subprocess.run(["nvcc", "-std=c++17", "-O0", "-Xcicc", "-O0", "-Xcompiler", "-fPIC,-O0", "-shared", "--threads", "0",
                    "-gencode", "arch=compute_100a,code=compute_100a", *defines, "-I", build.ROOT + "/include",
                    "-I", build.CSRC, "-o", out, *build.sources()], check=True, capture_output=True)
    lib = C.CDLL(out)
    f = lib.ssa_decode_attn_sparse
    f.restype, f.argtypes = C.c_int32, ssa.lib.ssa_decode_attn_sparse.argtypes

    def call(library, H, rows):
        d = good_desc()
        d.B, d.H, d.H_kv, d.max_ctx = 1, H, H, 2000
        one_each = sum((H * 4 * n + 255) // 256 * 256 for n in (128, 2))
        return library(C.byref(d), P, P, P, P, P, rows, P, rows, P, NUL, P, one_each, NUL, NUL)

    assert call(f, 200, 512) == ssa.ERR_CUDA
    assert call(f, 200, 1000) == ssa.ERR_WORKSPACE
    assert call(f, 74, 1000) == ssa.ERR_CUDA              # one block per two SMs: room for large ones
    assert call(ssa.lib.ssa_decode_attn_sparse, 200, 1000) == ssa.ERR_CUDA
