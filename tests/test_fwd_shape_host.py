"""The rule by which heads share a query tile of the attention forward, compiled for the host."""
import ctypes as C
import random
import subprocess

import pytest

from test_bwd_shape_host import CSRC, SMS


def compiled(folder):
    """pack_of(B, S, Hq, Hkv, dh, layers, causal): log2 of the heads that share a tile."""
    (folder / "r.cpp").write_text("""#include "kvp_fwd_shape.h"
extern "C" int pack_of(int B, int S, int Hq, int Hkv, int dh, int L, int causal) {
  return kvp::fwd_pack(kvp::FwdSizes{S, Hq / Hkv, dh, causal != 0, (long long)L * B * Hkv, %d});
}
""" % SMS)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, str(folder / "r.cpp"), "-o", str(folder / "r.so")], check=True)
    return C.CDLL(str(folder / "r.so")).pack_of


@pytest.fixture(scope="module")
def pack_of(tmp_path_factory):
    return compiled(tmp_path_factory.mktemp("fwd"))


def test_heads_stay_by_themselves_where_nothing_is_gained(pack_of):
    assert pack_of(1, 300, 16, 4, 64, 1, 1) == 0      # 20 items instead of 32, and longer ones
    assert pack_of(2, 512, 32, 8, 128, 2, 1) == 0
    assert pack_of(2, 8192, 32, 8, 128, 8, 1) == 0 and pack_of(4, 347, 32, 32, 128, 1, 1) == 0


@pytest.mark.parametrize("B,S,Hq,Hkv,dh,L,causal,packed", [
    (9, 2032, 64, 8, 128, 4, True, False),      # 2.33 ms whole heads, 2.78 packed
    (12, 1614, 64, 4, 128, 4, True, False),     # 2.20, 2.46
    (10, 1948, 128, 8, 128, 3, False, False),   # 7.49, 8.25
    (2, 1606, 16, 1, 64, 4, False, False),      # 135 us, 146
    (14, 117, 64, 8, 128, 4, True, False),      # 57, 63
    (2, 203, 64, 8, 128, 2, True, False),       # 13.9, 15.6: the fullest SM has one packed item more
    (6, 115, 64, 8, 64, 4, True, False),        # 22.7, 24.8
    (6, 1158, 128, 8, 64, 6, True, True),       # 2.01 ms, 1.67
    (3, 776, 16, 4, 64, 3, True, True),
    (10, 264, 16, 4, 128, 4, True, True),
])
def test_heads_are_packed_where_that_is_faster(pack_of, B, S, Hq, Hkv, dh, L, causal, packed):
    assert (pack_of(B, S, Hq, Hkv, dh, L, int(causal)) > 0) == packed


def test_a_tile_holds_heads_of_one_kv_head(pack_of):
    """The heads of a tile divide those of a KV head, as many as a power of two can, sixteen at most; none in sequences of more
    than 2048 tokens."""
    rng = random.Random(6)
    seen = set()
    for _ in range(4000):
        G, Hkv = rng.randint(1, 40), rng.randint(1, 8)
        S = int(2 ** rng.uniform(0, 13))
        pack = pack_of(rng.randint(1, 16), S, G * Hkv, Hkv, rng.choice((64, 128)), rng.randint(1, 8), rng.randint(0, 1))
        seen.add(pack)
        if pack:
            assert S <= 2048 and G % (1 << pack) == 0 and (pack == 4 or G % (2 << pack) != 0)
    assert seen == {0, 1, 2, 3, 4}
