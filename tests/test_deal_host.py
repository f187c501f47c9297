"""The rules by which a decode step's rows are dealt out to blocks, compiled for the host."""
import ctypes as C
import os
import random
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_15943_b200", "csrc")


@pytest.fixture(scope="module")
def deal(tmp_path_factory):
    d = tmp_path_factory.mktemp("deal")
    (d / "deal.cpp").write_text('#include "kvp_deal.h"\n'
                                'extern "C" int by_units(int d, long long t, long long u, long long l, int f) { return kvp::dealt_by_units(d, t, u, l, f); }\n'
                                'extern "C" int rest(int d, long long t, int f) { return kvp::unit_rest(d, t, f); }\n'
                                'extern "C" int shares(int d, int f, int m, long long p) { return kvp::shares_for(d, f, m, p); }\n')
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, str(d / "deal.cpp"), "-o", str(d / "deal.so")], check=True)
    lib = C.CDLL(str(d / "deal.so"))
    lib.by_units.argtypes = [C.c_int] + [C.c_longlong] * 3 + [C.c_int]
    lib.rest.argtypes, lib.shares.argtypes = [C.c_int, C.c_longlong, C.c_int], [C.c_int] * 3 + [C.c_longlong]
    return lib


FIT = {128: 296, 64: 592}     # blocks that fit on 148 SMs
ROUNDS = {128: 16, 64: 5}     # shares of a block that fits


def granules(lens):
    return [(n + 15) // 16 for n in lens]


def whole(deal, dh, lens, heads):
    g = granules(lens)
    return bool(deal.by_units(dh, sum(g) * heads, len(g) * heads, max(g), FIT[dh]))


@pytest.mark.parametrize("lens,heads", [([32768] + [300] * 63, 8), ([30000] + [200] * 39, 8), ([4096] * 4 + [64] * 28, 16), ([6000] * 2 + [100] * 30, 2)])
@pytest.mark.parametrize("dh", [64, 128])
def test_a_long_sequence_among_short_ones_is_cut(deal, dh, lens, heads):
    assert not whole(deal, dh, lens, heads)


@pytest.mark.parametrize("dh", [64, 128])
def test_no_block_gets_much_more_than_an_equal_share(deal, dh):
    rng = random.Random(3)
    for _ in range(2000):
        heads = rng.choice((1, 2, 8, 32, 64))
        lens = [int(2 ** rng.uniform(0, rng.uniform(1, 17))) for _ in range(rng.randint(1, 100))]
        g = granules(lens)
        if whole(deal, dh, lens, heads):
            assert max(g) <= max(8192 // dh, 2 * sum(g) * heads / FIT[dh])


@pytest.mark.parametrize("dh", [64, 128])
def test_a_full_table_of_short_units_stays_dealt_by_units(deal, dh):
    """The host decides by a table's capacity alone that no pieces can arise; the blocks must agree at any lengths."""
    rng = random.Random(4)
    for _ in range(2000):
        cap, B, heads = rng.randint(1, 140), rng.randint(1, 100), rng.choice((1, 2, 8, 32))
        if deal.by_units(dh, cap * B * heads, B * heads, cap, FIT[dh]):
            assert whole(deal, dh, [rng.randint(1, 16 * cap) for _ in range(B)], heads)


@pytest.mark.parametrize("dh", [64, 128])
def test_shares_grow_with_the_list_and_hold_work(deal, dh):
    fit = FIT[dh]
    n = [deal.shares(dh, fit, ROUNDS[dh] * fit, t) for t in range(0, 16000000, 997)]
    assert n == sorted(n) and n[0] == 1 and n[-1] % fit == 0 and n[-1] <= ROUNDS[dh] * fit


@pytest.mark.parametrize("dh", [64, 128])
def test_shares_cover_every_unit(deal, dh):
    """The kernels' dealing, restated: shares of the list with its empty places hold every granule once, and the merge finds
    the pieces of a unit between the shares of its first and its last granule."""
    rng = random.Random(5)
    fit = FIT[dh]
    for _ in range(60):
        lens = [int(2 ** rng.uniform(0, rng.uniform(1, 15))) for _ in range(rng.randint(1, 20))] * 4
        g = granules(lens)
        if whole(deal, dh, lens, 4):
            continue
        units = [n for n in g for _ in range(4)]
        rest = deal.rest(dh, sum(units), fit)
        places = sum(units) + rest * len(units)
        n = deal.shares(dh, fit, ROUNDS[dh] * fit, places)
        q, r = divmod(places, n)
        begin = [i * q + min(i, r) for i in range(n + 1)]
        assert q >= 1
        at, i = 0, 0
        for u in units:
            held = []
            while i < n and begin[i + 1] <= at:
                i += 1
            j = i
            while j < n and begin[j] < at + u:
                held.append(max(0, min(begin[j + 1], at + u) - max(begin[j], at)))
                j += 1
            assert sum(held) == u and min(held) > 0     # every share between the first and the last has a piece
            at += u + rest
