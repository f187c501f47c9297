"""The rules by which the attention backward is cut into CTAs and ordered, compiled for the host."""
import ctypes as C
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_15943_b200", "csrc")
SMS = 148


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("bwd")
    (d / "r.cpp").write_text("""#include "kvp_bwd_shape.h"
using namespace kvp;
static BwdSizes sizes(int B, int S, int Hq, int Hkv, int causal) { return BwdSizes{(S + 127) / 128, (S + 63) / 64, B * Hkv, Hq / Hkv, causal != 0, 148}; }
extern "C" int longest_first(int B, int S, int Hq, int Hkv, int dh, int L, int causal) {
  const BwdSizes z = sizes(B, S, Hq, Hkv, causal);
  return bwd_longest_first(z, L, bwd_steps_per_sm(z, L), (long long)B * S * Hq, dh);
}
extern "C" void cut(int B, int S, int Hq, int Hkv, int causal, int L, int* out) {
  const BwdSizes z = sizes(B, S, Hq, Hkv, causal);
  out[0] = bwd_target_steps(bwd_steps_per_sm(z, L));
  const BwdCut c = bwd_cut(z, L * z.G, out[0]);
  out[1] = c.window;
  out[2] = c.parts;
}
""")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, str(d / "r.cpp"), "-o", str(d / "r.so")], check=True)
    return C.CDLL(str(d / "r.so"))


@pytest.mark.parametrize("shape,first", [
    ((3, 776, 16, 4, 64, 3, 1), True),        # 57 MB: order costs no L2 locality
    ((1, 4096, 8, 8, 128, 1, 1), True),
    ((8, 1024, 32, 8, 128, 4, 1), False),     # 1.1 GB
    ((2, 4096, 32, 8, 128, 4, 1), False),
    ((1, 1024, 16, 4, 64, 4, 0), True),
    ((1, 4096, 16, 4, 128, 1, 0), False),     # no mask: 67 MB, but 221 steps per SM
    ((4, 2048, 32, 32, 128, 1, 0), False),
    ((2, 8192, 8, 8, 64, 1, 1), False),       # 67 MB, but 450 steps per SM
])
def test_order(rules, shape, first):
    assert bool(rules.longest_first(*shape)) == first


@pytest.mark.parametrize("B,S,Hq,Hkv,causal,L", [(1, 64, 4, 2, 1, 1), (2, 128, 4, 2, 1, 4), (1, 1024, 16, 4, 0, 1), (3, 776, 16, 4, 1, 3), (2, 8192, 32, 8, 1, 4)])
def test_every_stream_and_query_tile_is_in_a_cta(rules, B, S, Hq, Hkv, causal, L):
    out = (C.c_int * 3)()
    rules.cut(B, S, Hq, Hkv, causal, L, out)
    streams, n_qt = L * Hq // Hkv, (S + 63) // 64
    assert 1 <= out[1] <= n_qt and 1 <= out[2] <= streams
    if S <= 128:
        assert out[2] <= (1 if out[1] < n_qt else 2)     # at most two terms: results do not differ from run to run
