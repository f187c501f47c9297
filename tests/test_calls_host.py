"""The native calls of the binding hand the library what its ctypes path does, and leave everything unusual to that path."""
import ctypes as C
import os
import subprocess
import sys
import types

import pytest
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NAMES = ("gemm", "rmsnorm", "rope", "swiglu", "add", "proj_fwd", "proj_bwd", "out_proj_fwd", "out_proj_bwd", "attn_fwd", "attn_bwd",
         "cache_append", "decode")
# arguments of the entry points: i integer, l 64-bit integer, f float, p pointer, S structure, D donor map, A array of pointers
FORMS = {"gemm": "iiiplipliplip", "rmsnorm": "iippfpp", "rope": "iiiifipp", "swiglu": "lpppp", "add": "lpppp",
         "proj_fwd": "SDAAAAAAAplp", "proj_bwd": "SDAAAAAAAAAAAplp", "out_proj_fwd": "SAAAp", "out_proj_bwd": "SAAAAAp",
         "attn_fwd": "SDifAAAAAplp", "attn_bwd": "SDifAAAAAAAAAplp", "cache_append": "SDAAAAppp", "decode": "SDfAAAppAAiiplp"}
TYPES = dict(i=C.c_int, l=C.c_int64, f=C.c_float, p=C.c_void_p, S=C.c_void_p, D=C.c_void_p, A=C.c_void_p)


@pytest.fixture
def record(monkeypatch):
    """What reaches the library, by either path: (name, arguments with the arrays read out)."""
    from paper_2608_15943_b200 import kvp
    seen, keep = [], []

    def make(name):
        form = FORMS[name]
        size = C.sizeof(kvp.DecodeDesc if name in ("cache_append", "decode") else kvp.Shape)

        def called(*args):
            layers = C.cast(args[0], C.POINTER(C.c_int32))[0] if form[0] == "S" else 0
            read = {"S": lambda v: C.string_at(v, size), "D": lambda v: C.string_at(v, 4 * layers), "A": lambda v: C.string_at(v, 8 * layers)}
            seen.append((name, [read.get(k, lambda v: v)(v) for k, v in zip(form, args)]))
            return 0
        return C.CFUNCTYPE(C.c_int, *[TYPES[k] for k in form])(called)
    for name in NAMES:
        cb = make(name)
        keep.append(cb)
        monkeypatch.setattr(kvp.lib, "kvp_" + name, cb)
    real = kvp._pack
    original = [C.cast(getattr(C.CDLL(kvp.LIB_PATH), "kvp_" + n), C.c_void_p).value for n in NAMES]
    real.bind([C.cast(cb, C.c_void_p).value for cb in keep], kvp.Shape, kvp.DecodeDesc)
    monkeypatch.setattr(kvp, "_stream", lambda: 0x7f0000001238)
    none = types.SimpleNamespace(**{n: lambda *a: NotImplemented for n in NAMES})

    def both(call):
        """The arguments that `call` hands over through ctypes, and whether the native path took it (with the same ones)."""
        del seen[:]
        monkeypatch.setattr(kvp, "_pack", none)
        call()
        taken = []
        spy = types.SimpleNamespace(**{n: (lambda n: lambda *a: taken.append(getattr(real, n)(*a)) or taken[-1])(n) for n in NAMES})
        monkeypatch.setattr(kvp, "_pack", spy)
        call()
        monkeypatch.setattr(kvp, "_pack", real)
        assert len(seen) == 2 and seen[0] == seen[1]
        return taken == [0]
    both.seen = seen
    yield kvp, both
    real.bind(original, kvp.Shape, kvp.DecodeDesc)


def bf(*shape):
    return torch.zeros(*shape, dtype=torch.bfloat16)


class Sub(torch.Tensor):
    pass


def test_single_operators(record):
    kvp, both = record
    a, b, c = bf(6, 16), bf(24, 16), bf(6, 24)
    for form in ((a, b, c), (a, b, c.float()), (bf(6, 40)[:, 8:24], bf(24, 32)[:, :16], bf(6, 64)[:, 8:32]), (bf(16, 6), b, c, True), (a, bf(16, 24), c, False, True),
                 (bf(16, 6), bf(16, 24), c, True, True), (a.t(), b, c)):
        assert both(lambda: kvp.gemm(*form))
    x, w, y = bf(5, 32), torch.nn.Parameter(bf(32)), bf(5, 32)
    assert both(lambda: kvp.rmsnorm(x, w, 1e-5, y))
    for t in (bf(2, 3, 4, 64), bf(2, 3, 8, 64)[:, 1:, :4]):
        assert both(lambda: kvp.rope(t)) and both(lambda: kvp.rope(t, 500000.0, 77))
    for f in (kvp.add, kvp.swiglu):
        for t in (bf(3, 8), bf(24), bf(0), bf(2, 3, 4)[1], torch.zeros(())):
            assert both(lambda: f(t, t, t))
    # left to ctypes: subclasses, other kinds of numbers
    s, flat, small = bf(6, 16).as_subclass(Sub), bf(384), bf(1, 1, 1, 8)
    assert not both(lambda: kvp.gemm(s, b, c)) and not both(lambda: kvp.gemm(a, b, c, 0, 0)) and not both(lambda: kvp.gemm(a, flat, c))
    assert not both(lambda: kvp.rmsnorm(x, w, 1, x)) and not both(lambda: kvp.rope(small, 10000, 2)) and not both(lambda: kvp.add(s, s, s))


def test_layer_calls(record):
    kvp, both = record
    L = 3
    sh, de = kvp.Shape(L, 2, 5, 64, 4, 2, 64, kvp.F32), kvp.DecodeDesc(L, 2, 4, 2, 64, 16, 3, 7)
    donor, t, ws = [0, 1, 1], lambda: [bf(2), None, bf(3, 4)[1:]], bf(100)
    kinds = (lambda x: x, tuple)
    for kind in kinds:
        arr = [kind(t()) for _ in range(11)]
        dm = kind(donor)
        assert both(lambda: kvp.proj_fwd(sh, dm, *arr[:7])) and both(lambda: kvp.proj_fwd(sh, dm, *arr[:7], ws))
        assert both(lambda: kvp.proj_bwd(sh, dm, *arr, ws))
        assert both(lambda: kvp.out_proj_fwd(sh, *arr[:3])) and both(lambda: kvp.out_proj_bwd(sh, *arr[:5]))
        for more in ({}, dict(causal=False, scale=0.5, ws=ws)):
            assert both(lambda: kvp.attn_fwd(sh, dm, *arr[:5], **more))
        for more in ({}, dict(causal=False, scale=0.25)):
            assert both(lambda: kvp.attn_bwd(sh, dm, *arr[:9], ws, **more))
        table, lengths = torch.zeros(2, 3, dtype=torch.int32), torch.ones(2, dtype=torch.int32)
        assert both(lambda: kvp.cache_append(de, dm, *arr[:4], table, lengths))
        for more in ({}, dict(scale=0.125, layer_begin=1), dict(layer_end=2), dict(layer_begin=1, layer_end=3)):
            assert both(lambda: kvp.decode(de, dm, *arr[:3], table, lengths, *arr[3:5], ws, **more))
    arr = [t() for _ in range(11)]
    odd = [t()[:2] + [bf(4).as_subclass(Sub)]] + arr[1:]
    assert not both(lambda: kvp.proj_fwd(sh, donor, *odd[:7])) and not both(lambda: kvp.attn_fwd(sh, donor, *odd[:5]))
    assert not both(lambda: kvp.proj_fwd(sh, torch.tensor(donor), *arr[:7])) and not both(lambda: kvp.attn_fwd(sh, [0, True, 1], *arr[:5], causal=1, scale=0))
    assert not both(lambda: kvp.decode(de, donor, *arr[:3], table, lengths, *arr[3:5], ws, scale=0))


def test_short_lists(record):
    """What a list lacks of its L entries reaches the library as null pointers, never as entries of the next list."""
    kvp, both = record
    L = 4
    sh, de, ws = kvp.Shape(L, 2, 5, 64, 4, 2, 64), kvp.DecodeDesc(L, 2, 4, 2, 64, 16, 3, 7), bf(100)
    donor, table = [0, 1, 1, 1], torch.zeros(2, 3, dtype=torch.int32)

    def arrays(short, n):
        a = [[bf(2) for _ in range(L)] for _ in range(11)]
        a[short] = a[short][:n]
        return a

    def passed(call, at, entries):
        """`call` hands over, as its array number `at`, the tensors of `entries` and nulls behind them."""
        want = b"".join(t.data_ptr().to_bytes(8, "little") for t in entries)
        assert both(call)
        name, args = both.seen[0]
        got = [v for kind, v in zip(FORMS[name], args) if kind == "A"][at]
        assert got == want + bytes(8 * L - len(want))
    for n in (0, 1, 3):
        for i in range(11):
            a = arrays(i, n)
            passed(lambda: kvp.proj_bwd(sh, donor, *a, ws), i, a[i])
            if i < 9:
                passed(lambda: kvp.attn_bwd(sh, donor, *a[:9], ws), i, a[i])
            if i < 7:
                passed(lambda: kvp.proj_fwd(sh, donor, *a[:7]), i, a[i])
            if i < 5:
                passed(lambda: kvp.attn_fwd(sh, donor, *a[:5]), i, a[i])
                passed(lambda: kvp.decode(de, donor, *a[:3], table, table, *a[3:5], ws), i, a[i])
            if i < 4:
                passed(lambda: kvp.cache_append(de, donor, *a[:4], table, table), i, a[i])
    sh, a = kvp.Shape(2, 1, 8, 64, 1, 1, 64), [[bf(2) for _ in range(2)] for _ in range(5)]
    for i in range(5):                           # without a donor map: one null, at which the entry points stop
        b = a[:i] + [a[i][:1]] + a[i + 1:]
        for call, lists in ((kvp.out_proj_fwd, 3), (kvp.out_proj_bwd, 5)):
            if i < lists:
                assert both(lambda: call(sh, *b[:lists]))
                assert both.seen[0][1][1 + i] == b[i][0].data_ptr().to_bytes(8, "little") + bytes(8)


@pytest.mark.parametrize("native", [True, False])
def test_short_lists_refused(native, monkeypatch):
    """By the library itself, before it launches anything."""
    from paper_2608_15943_b200 import kvp
    if not native:
        monkeypatch.setattr(kvp, "_pack", types.SimpleNamespace(**{n: lambda *a: NotImplemented for n in NAMES}))
    x, table = bf(64, 64), torch.zeros(2, 3, dtype=torch.int32)
    sh, de = kvp.Shape(2, 1, 64, 64, 1, 1, 64), kvp.DecodeDesc(2, 2, 1, 1, 64, 16, 3, 7)
    full, one, ws = [x, x], [x], bf(1 << 23)

    def refused(call, status):
        with pytest.raises(kvp.KvpError) as e:
            call()
        assert e.value.status == status
    calls = ((lambda d, *a: kvp.proj_fwd(sh, d, *a, ws), 7), (lambda d, *a: kvp.proj_bwd(sh, d, *a, ws), 11), (lambda d, *a: kvp.proj_bwd(sh, d, *a, ws, 0, 1), 11),
             (lambda d, *a: kvp.attn_fwd(sh, d, *a, ws=ws), 5), (lambda d, *a: kvp.attn_bwd(sh, d, *a, ws), 9),
             (lambda d, *a: kvp.cache_append(de, d, *a, table, table), 4), (lambda d, *a: kvp.decode(de, d, *a[:3], table, table, *a[3:], ws), 5),
             (lambda d, *a: kvp.decode_static(de, d, *a[:3], table, table, *a[3:]), 5))
    for call, lists in calls:
        refused(lambda: call([0], *[full] * lists), kvp.ERR_BAD_DONOR)
        if call is calls[-1][0]:
            continue      # (looks for its scratch on the device first)
        for i in range(lists):
            refused(lambda: call([0, 1], *[one if j == i else full for j in range(lists)]), kvp.ERR_INVALID_ARG)
    for call, lists in ((kvp.out_proj_fwd, 3), (kvp.out_proj_bwd, 5)):
        for i in range(lists):
            refused(lambda: call(sh, *[one if j == i else full for j in range(lists)]), kvp.ERR_INVALID_ARG)
    assert kvp.workspace_bytes(kvp.OP_ATTN_BWD, sh, [0]) == 0 and kvp.decode_workspace_bytes(de, [0]) == 0


def test_many_layers(record):
    """More entries than the native path has room for."""
    kvp, both = record
    for L, native in ((60, True), (256, False), (300, False)):
        sh, ws = kvp.Shape(L, 1, 1, 64, 1, 1, 64), bf(1)
        arr = [[ws] * L] * 11
        assert both(lambda: kvp.proj_bwd(sh, [0] * L, *arr, ws)) == native


def test_refused_as_before():
    """What ctypes refuses, and how, with the library itself."""
    from paper_2608_15943_b200 import kvp
    x = bf(4, 8)
    for call, err in ((lambda: kvp.add(x, x, None), AttributeError), (lambda: kvp.gemm(x, x, bf(4)), ValueError), (lambda: kvp.rope(x), ValueError),
                      (lambda: kvp.attn_fwd(kvp.Shape(1, 1, 1, 64, 1, 1, 64), [2**31], *[[x]] * 5), OverflowError),
                      (lambda: kvp.attn_fwd(kvp.DecodeDesc(1, 1, 1, 1, 64, 16, 1, 1), [0], *[[x]] * 5), C.ArgumentError),
                      (lambda: kvp.rmsnorm(x, x, "x", x), ValueError)):
        with pytest.raises(err):
            call()
    with pytest.raises(kvp.KvpError) as e:
        kvp.add(bf(3), bf(3), bf(3))
    assert e.value.status == kvp.ERR_UNSUPPORTED and "kvp_add" in str(e.value)


THROWS = """
#include <new>
#include <stdexcept>
int calls = 0;
extern "C" int count() { return calls; }
extern "C" int no_memory(long, void*, void*, void*, void*) { ++calls; throw std::bad_alloc(); }
extern "C" int error(long, void*, void*, void*, void*) { ++calls; throw std::runtime_error("of the library"); }
"""
CATCHES = """
import ctypes as C, sys, threading, torch
from paper_2608_15943_b200 import kvp
lib, x = C.CDLL(sys.argv[1]), torch.zeros(8, dtype=torch.bfloat16)
for n, (name, kind) in enumerate((("no_memory", MemoryError), ("error", RuntimeError))):
    kvp._pack.bind([C.cast(getattr(lib, name), C.c_void_p).value] * 13, kvp.Shape, kvp.DecodeDesc)
    try:
        kvp.add(x, x, x)
    except kind as e:
        assert name == "no_memory" or "of the library" in str(e)
    else:
        raise AssertionError(name)
    assert lib.count() == n + 1
    t = threading.Thread(target=lambda: sum(range(1000)))   # the interpreter's lock is held, and can be handed on
    t.start()
    t.join()
"""


def test_exceptions_of_the_library(tmp_path):
    """An exception out of an entry point reaches Python; the entry point is not called again."""
    (tmp_path / "throws.cpp").write_text(THROWS)
    subprocess.run(["g++", "-shared", "-fPIC", "-o", str(tmp_path / "throws.so"), str(tmp_path / "throws.cpp")], check=True)
    done = subprocess.run([sys.executable, "-c", CATCHES, str(tmp_path / "throws.so")], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert done.returncode == 0, done.stderr
