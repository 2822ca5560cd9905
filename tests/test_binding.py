"""binding/ssa_call.c: every argument of a Python call reaches the parameter of the C entry point that it stands for.  The
entry points are Python callbacks with the C signatures, so nothing here needs a GPU."""
import ctypes as C
import importlib.util
import sysconfig
import types

import numpy as np
import pytest
import torch

from paper_2404_09336_b200 import build, ssa

TABLES = [f"table{i}" for i in range(9)]
# name: the call's arguments, and the entry point's as they should arrive ("#x" elements, "/x" row stride, "*x" bytes of x)
CALLS = {
    "spans_to_index": ("offs spans ctx idx cnt status 7", "offs spans ctx #ctx idx /idx cnt status 7"),
    "decode_attn_sparse": ("desc q k v ctx idx cnt 11 out lse ws status 7",
                           "desc q k v ctx idx /idx cnt 11 out lse ws *ws status 7"),
    "decode_attn_spans": ("desc q k v ctx offs spans 5 11 out lse idx cnt ws status 7",
                          "desc q k v ctx offs spans 5 11 out lse idx /idx cnt ws *ws status 7"),
    "decode_attn_sparse_multiq": ("desc 3 64 65 q k v ctx idx cnt 11 out lse ws status 7",
                                  "desc 3 64 65 q k v ctx idx /idx cnt 11 out lse ws *ws status 7"),
    "decode_attn_dense_multiq": ("desc 3 64 65 q k v ctx out lse ws status 7", "desc 3 64 65 q k v ctx out lse ws *ws status 7"),
    "spans_to_blockmask": ("offs spans ctx 32 idx mask cnt status 7", "offs spans ctx #ctx 32 idx mask /idx cnt status 7"),
    "decode_attn_blockmask": ("desc q k v ctx idx mask cnt 32 9 out lse ws status 7",
                              "desc q k v ctx idx mask /idx cnt 32 9 out lse ws *ws status 7"),
    "decode_attn_sparse_paged": ("desc q k v paging ctx idx cnt 11 out lse ws status 7",
                                 "desc q k v paging ctx idx /idx cnt 11 out lse ws *ws status 7"),
    "decode_attn_dense_paged": ("desc q k v paging ctx out lse ws status 7", "desc q k v paging ctx out lse ws *ws status 7"),
    "refs_to_index": (" ".join(TABLES) + " idx cnt status 7", "tables #table8 idx /idx cnt status 7"),
    "refs_to_spans": (" ".join(TABLES) + " offs spans 9 status 7", "tables #table8 offs spans 9 status 7"),
    "decode_step": ("desc step 7", "desc step 7"),
    "decode_attn_sparse_noalloc": ("desc q k v ctx idx cnt 11 out lse status 7", "desc q k v ctx idx /idx cnt 11 out lse status 7"),
    "decode_attn_dense": ("desc q k v ctx out lse ws status 7", "desc q k v ctx out lse ws *ws status 7"),
}


def bound():
    """A second instance of the module, bound to callbacks that keep what they were given."""
    spec = importlib.util.spec_from_file_location("apart._ssa_call", build.build_binding())
    module = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(module)
    got, keep, addresses = {}, [], {}
    for name in CALLS:
        f = getattr(ssa.lib, "ssa_" + name)
        types = [C.c_void_p if t.__name__.startswith("LP_") else t for t in f.argtypes]

        def entry(*args, name=name):
            got[name] = list(args)
            if name.startswith("refs"):
                t = C.cast(args[0], C.POINTER(ssa.AnchorTables)).contents
                got[name][0] = [getattr(t, f) for f, _ in t._fields_]
            return 3
        keep.append(C.CFUNCTYPE(C.c_int32, *types)(entry))
        addresses["ssa_" + name] = C.cast(keep[-1], C.c_void_p).value
    module.bind(addresses)
    return module, got, keep


def values(rows):
    i32 = lambda *s: torch.zeros(s, dtype=torch.int32)
    d = {n: torch.zeros(4, 2, dtype=torch.bfloat16) for n in ("q", "k", "v", "out", "lse")}
    d.update(offs=i32(4), spans=i32(3, 9, 2), ctx=i32(rows), cnt=i32(rows), status=i32(1), mask=i32(rows, 8), ws=torch.zeros(321),
             idx=i32(rows, 2, 40)[:, 1, :36], desc=ssa.AttnDesc(), paging=ssa.Paging(), step=ssa.Step())
    d.update({n: i32(5 + i) for i, n in enumerate(TABLES)})
    return d


@pytest.mark.parametrize("rows", [1, 3])
@pytest.mark.parametrize("name", sorted(CALLS))
def test_arguments_arrive(name, rows):
    module, got, _ = bound()
    d = values(rows)
    at = lambda x: C.addressof(x) if isinstance(x, C.Structure) else x.data_ptr()

    def want(word):
        if word == "tables":
            return [at(d[n]) for n in TABLES]
        if word[0] == "#":
            return d[word[1:]].numel()
        if word[0] == "/":
            return 80 if rows > 1 else 36                # one row: its length, whatever the stride of that dimension
        if word[0] == "*":
            return 4 * 321
        return at(d[word]) if word in d else int(word)

    args, params = (w.split() for w in CALLS[name])
    assert getattr(module, name)(*(d[w] if w in d else int(w) for w in args)) == 3
    assert got[name] == [want(w) for w in params]
    # absent tensors are NULL with no bytes and no stride; numbers of other types are taken
    optional = {"lse", "ws", "status", "paging"} | ({"idx"} if "attn" in name else set())
    assert getattr(module, name)(*(None if w in optional else d[w] if w in d else np.int64(w) for w in args)) == 3
    assert got[name] == [(None if w in optional else 0 if w.strip("/*") in optional else want(w)) for w in params]


def test_wrong_arguments_raise_before_the_entry_point():
    module, got, _ = bound()
    d = values(3)
    good = [d[w] if w in d else int(w) for w in CALLS["decode_attn_dense"][0].split()]
    for i, bad, error in ((0, d["step"].host_in, TypeError), (0, ssa.Paging(), TypeError), (1, 5, AttributeError),
                          (7, "x", AttributeError), (9, "x", ValueError)):
        args = list(good)
        args[i] = bad
        with pytest.raises(error):
            module.decode_attn_dense(*args)
    with pytest.raises(TypeError):
        module.decode_attn_dense(*good[:-1])
    assert not got
    # another library's binding in the same process is its own
    assert ssa.decode_attn_dense(d["desc"], None, None, None, None, None, stream=0, check=False) == ssa.ERR_NULL


class _Longer(ssa.AttnDesc):
    _fields_ = [("note", C.c_int64)]


def test_only_the_descriptor_s_own_class_is_taken():
    """Null tensors: a call that gets past its descriptor is refused by the library, not by the binding."""
    tail = (None,) * 8 + (0,)
    big = type("Big", (C.Structure,), {"_fields_": [("x", C.c_char * 400)]})()
    for wrong in (ssa.Step(), ssa.Paging(), big, bytes(400), bytearray(112), np.zeros(14, np.int64), None, 5):
        with pytest.raises(TypeError, match="ssa_attn_desc"):
            ssa._call.decode_attn_dense(wrong, *tail)
        if wrong is not None:
            with pytest.raises(TypeError, match="ssa_paging"):
                if isinstance(wrong, ssa.Paging):
                    wrong = ssa.AttnDesc()
                ssa._call.decode_attn_dense_paged(ssa.AttnDesc(), None, None, None, wrong, *tail[3:])
    for wrong in (ssa.AttnDesc(), bytes(400), big):
        with pytest.raises(TypeError, match="ssa_step"):
            ssa._call.decode_step(ssa.AttnDesc(), wrong, 0)
    for right in (ssa.AttnDesc(), _Longer()):
        assert ssa._call.decode_attn_dense(right, *tail) == ssa.ERR_NULL
    # bound without classes: a buffer of the exact size
    module, got, _ = bound()
    for wrong in (ssa.Step(), bytes(C.sizeof(ssa.AttnDesc) + 1)):
        with pytest.raises(TypeError):
            module.decode_attn_dense(wrong, *tail)
    assert not got and module.decode_attn_dense(ssa.AttnDesc(), *tail) == 3


def test_each_interpreter_has_a_binding_of_its_own():
    assert build.BINDING.endswith(sysconfig.get_config_var("EXT_SUFFIX")) and ssa._call.__file__ == build.BINDING


def test_calls_go_through_ctypes_where_the_binding_cannot_be_built(monkeypatch):
    """A finished library, no compiler: the import warns, and every argument arrives as through the binding."""
    def no_compiler():
        raise RuntimeError("gcc not found")
    monkeypatch.setattr(build, "build_binding", no_compiler)
    with pytest.warns(RuntimeWarning, match="gcc not found"):
        calls = ssa._load_calls()
    assert calls.decode_attn_dense(ssa.AttnDesc(), *(None,) * 8, 0) == ssa.ERR_NULL
    with pytest.raises((TypeError, C.ArgumentError)):
        calls.decode_attn_dense(ssa.Step(), *(None,) * 8, 0)
    monkeypatch.undo()
    module, got, keep = bound()
    through = ssa._CtypesCalls(types.SimpleNamespace(**{"ssa_" + name: f for name, f in zip(CALLS, keep)}))
    optional = {"lse", "ws", "status", "paging"}
    for rows in (1, 3):
        d = values(rows)
        for name, (args, _) in CALLS.items():
            for absent in (set(), optional | ({"idx"} if "attn" in name else set())):
                given = [None if w in absent else d[w] if w in d else int(w) for w in args.split()]
                assert getattr(module, name)(*given) == 3
                want = got.pop(name)
                assert getattr(through, name)(*given) == 3 and got.pop(name) == want, name
