"""Whether outputs of a call share memory with its inputs, compiled for the host."""
import ctypes as C
import os
import random
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_15943_b200", "csrc")


@pytest.fixture(scope="module")
def shares(tmp_path_factory):
    d = tmp_path_factory.mktemp("overlap")
    (d / "r.cpp").write_text("""#include "kvp_overlap.h"
extern "C" int shares(int L, const void* const* a, size_t na, const int32_t* da, const void* const* b, size_t nb, const int32_t* db, int same_layer) {
  const kvp::Tensors out{a, na, da};
  return kvp::Outputs(L, {out}).meet(kvp::Tensors{b, nb, db}, same_layer ? &out : nullptr);
}
""")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, str(d / "r.cpp"), "-o", str(d / "r.so")], check=True)
    lib = C.CDLL(str(d / "r.so"))

    def call(a, na, da, b, nb, db, same_layer=False):
        arr = lambda xs: (C.c_void_p * len(xs))(*xs)
        ints = lambda xs: None if xs is None else (C.c_int32 * len(xs))(*xs)
        return bool(lib.shares(len(a), arr(a), C.c_size_t(na), ints(da), arr(b), C.c_size_t(nb), ints(db), int(same_layer)))
    return call


def test_edges(shares):
    assert shares([100], 10, None, [109], 1, None) and shares([100], 10, None, [91], 10, None) and shares([100], 10, None, [90], 30, None)
    assert not shares([100], 10, None, [110], 10, None) and not shares([100], 10, None, [90], 10, None)
    a, b = [100, 0], [400, 0]                       # the consumers' entries are no tensors, null or not
    assert not shares(a, 10, [0, 0], b, 10, [0, 0]) and not shares([100, 400], 10, [0, 0], [400, 100], 10, [0, 0])
    assert shares([100, 400], 10, None, [400, 100], 10, [0, 0]) and not shares([100, 0], 10, [0, 0], [0, 300], 10, None)

    assert not shares([100, 200], 10, None, [100, 200], 10, None, True) and shares([100, 200], 10, None, [100, 206], 10, None, True)
    assert shares([100, 200], 10, None, [200, 100], 10, None, True)


def test_any(shares):
    rng = random.Random(5)
    found = 0
    for _ in range(400):
        L = rng.randint(1, 6)
        na, nb = rng.randint(1, 30), rng.randint(1, 30)
        a, b = [x * na for x in rng.sample(range(40, 40 + 400 // na), L)], [rng.randrange(40 * na, 40 * na + 400) for _ in range(L)]   # outputs apart
        da, db = (rng.choice((None, [rng.choice((l, 0)) for l in range(L)])) for _ in range(2))
        tensors = lambda xs, d: [x for l, x in enumerate(xs) if d is None or d[l] == l]
        want = any(set(range(x, x + na)) & set(range(y, y + nb)) for x in tensors(a, da) for y in tensors(b, db))
        found += want
        assert shares(a, na, da, b, nb, db) == want
    assert 50 < found < 350
