"""The rules by which a forward GEMM chooses its kernel and tiles, compiled for the host."""
import ctypes as C
import os
import random
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_15943_b200", "csrc")
SMS = 148
SINGLE, PAIR, TALL, SPLIT = range(4)


def compiled(folder):
    """choose(list of (M, N, K)) -> (kernel, tokens per tile, K split)."""
    (folder / "c.cpp").write_text("""#include "kvp_gemm_choice.h"
using namespace kvp;
extern "C" void choose(const int* mnk, int n, int* out) {
  GemmSize g[32];
  int rows = 0;
  for (int i = 0; i < n; ++i) {
    g[i] = GemmSize{mnk[3 * i], mnk[3 * i + 1], mnk[3 * i + 2]};
    rows = std::max(rows, g[i].M);
  }
  if (rows <= SPLIT_MAX_ROWS) {
    const SplitConfig c = split_config(g, n, 148);
    out[0] = Choice::kSplit, out[1] = c.nt, out[2] = c.split;
  } else if (rows > CHOICE_MAX_ROWS) {
    out[0] = Choice::kPair, out[1] = 0, out[2] = 1;
  } else {
    const Choice c = choose_forward(g, n, 148);
    out[0] = c.kind, out[1] = c.nt, out[2] = c.split;
  }
}
""")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, str(folder / "c.cpp"), "-o", str(folder / "c.so")], check=True)
    lib = C.CDLL(str(folder / "c.so"))

    def choose(problems):
        out, flat = (C.c_int * 3)(), [x for p in problems for x in p]
        lib.choose((C.c_int * len(flat))(*flat), len(problems), out)
        return tuple(out)
    return choose


@pytest.fixture(scope="module")
def choose(tmp_path_factory):
    return compiled(tmp_path_factory.mktemp("choice"))


def some_lists(seed, n=3000):
    rng = random.Random(seed)
    for _ in range(n):
        M = int(2 ** rng.uniform(0, 12))
        yield [(M, 8 * rng.randint(1, 4000 if rng.random() < 0.3 else 512), 8 * int(2 ** rng.uniform(0, 11))) for _ in range(rng.choice((1, 1, 2, 5)))]


def test_every_cta_of_a_split_has_k_blocks(choose):
    """Problems of different depth in one launch: the shallowest bounds the split, an empty range would add whatever the
    accumulator held."""
    for problems in some_lists(1):
        kind, nt, split = choose(problems)
        if kind == SPLIT:
            assert split <= min((k + 63) // 64 for _, _, k in problems), problems
            assert 16 <= nt <= 256 and nt % 16 == 0


def test_pair_tiles_go_in_steps_of_32_tokens(choose):
    """The N of an MMA of M = 256 on a CTA pair; the kernel's remainders use the same unit."""
    seen = 0
    for problems in some_lists(2):
        kind, nt, _ = choose(problems)
        if kind == TALL:
            seen += 1
            assert 32 <= nt <= 256 and nt % 32 == 0, problems
    assert seen > 300
    source = open(os.path.join(CSRC, "kvp_gemm.cu")).read()
    assert "unit = g.a_mn ? 128 : TALL_UNIT" in source
