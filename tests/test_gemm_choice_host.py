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
    """choose(list of (M, N, K)) -> (kernel, tokens per tile, K split); and, up to 128 rows, split_choice(the same) ->
    (tokens per tile, CTAs of a cluster, accumulators of a CTA, stages)."""
    (folder / "c.cpp").write_text("""#include "kvp_gemm_choice.h"
using namespace kvp;
extern "C" void split_choice(const int* mnk, int n, int* out) {
  GemmSize g[32];
  for (int i = 0; i < n; ++i) g[i] = GemmSize{mnk[3 * i], mnk[3 * i + 1], mnk[3 * i + 2]};
  const SplitConfig c = split_config(g, n, 148);
  out[0] = c.nt, out[1] = c.split, out[2] = c.parts, out[3] = c.stages;
}
extern "C" int streams(const int* mnk, int n) {
  GemmSize g[32];
  for (int i = 0; i < n; ++i) g[i] = GemmSize{mnk[3 * i], mnk[3 * i + 1], mnk[3 * i + 2]};
  return stream_weights(g, n, split_config(g, n, 148).nt);
}
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

    def caller(f, size):
        def call(problems):
            out, flat = (C.c_int * size)(), [x for p in problems for x in p]
            f((C.c_int * len(flat))(*flat), len(problems), out)
            return tuple(out)
        return call
    def streams(problems):
        flat = [x for p in problems for x in p]
        return bool(lib.streams((C.c_int * len(flat))(*flat), len(problems)))
    return caller(lib.choose, 3), caller(lib.split_choice, 4), streams


@pytest.fixture(scope="module")
def choices(tmp_path_factory):
    return compiled(tmp_path_factory.mktemp("choice"))


@pytest.fixture(scope="module")
def choose(choices):
    return choices[0]


@pytest.mark.parametrize("problems,streamed", [
    ([(1, 4096, 4096)], True), ([(128, 4096, 4096)], True), ([(16, 4096, 4088)], False),    # 32 MB and a little less
    ([(8, 4096, 2048), (8, 1024, 2048), (8, 1024, 2048)], False), ([(8, 4096, 4096), (8, 1024, 4096), (8, 1024, 4096)], True),
    ([(8, 4096, 4096), (160, 4096, 4096)], False), ([(129, 11008, 4096)], False),           # more rows than one tile, than 128
    ([(5, 4104, 4104)], True), ([(128, 11016, 1608)], True), ([(33, 18440, 920)], True), ([(70, 1032, 16400)], True),   # (those of the GPU's test)
])
def test_streamed_weights(choices, problems, streamed):
    assert choices[2](problems) == streamed


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


def test_bounds_of_the_few_rows_kernel(choices):
    """What its launch and its blocks rely on: tokens per tile an MMA can have, a ring of two stages or more, accumulators
    that fit tensor memory and sums that fit shared memory, half of both where CTAs share an SM."""
    seen = set()
    for problems in some_lists(3, 6000):
        problems = [((m - 1) % 128 + 1, n, k) for m, n, k in problems]
        nt, split, parts, stages = choices[1](problems)
        seen.add((split, parts))
        rows = max(m for m, _, _ in problems)
        ctas = sum((n + 127) // 128 * ((m + nt - 1) // nt) for m, n, _ in problems) * split
        assert 16 <= nt <= 128 and nt % 16 == 0 and nt < rows + 16
        assert split in (1, 2, 4, 8) and parts in (1, 2) and split * parts <= 8
        assert split == 1 or ctas < 2 * SMS, problems
        assert parts == 1 or split > 1 and ctas <= SMS
        ring = (220 if ctas <= SMS else 110) * 1024
        assert 2 <= stages <= 8 and stages * (16384 + nt * 128) <= ring and parts * nt * 512 <= ring, problems
        assert parts * max(nt, 32) <= (512 if ctas <= SMS else 256)
    assert seen == {(1, 1), (2, 1), (4, 1), (8, 1), (2, 2), (4, 2)}


def test_pieces_of_k_go_by_columns_and_depth(choices):
    """The smallest power of two that gives 128 tiles, two k-blocks in each: the same for any number of rows."""
    for problems in some_lists(4):
        columns, depth = sum((n + 127) // 128 for _, n, _ in problems), min((k + 63) // 64 for _, _, k in problems)
        pieces = 1
        while pieces < 8 and 2 * pieces <= depth and columns * pieces < 128:
            pieces *= 2
        for rows in (1, 16, 17, 64, 128):
            _, split, parts, _ = choices[1]([(rows, n, k) for _, n, k in problems])
            assert split * parts == pieces, (rows, problems)


@pytest.fixture(scope="module")
def deal(tmp_path_factory):
    folder = tmp_path_factory.mktemp("deal")
    (folder / "d.cpp").write_text("""#include "kvp_gemm_choice.h"
using namespace kvp;
extern "C" float tile_us(int kb, int nt, int f32) { return gradient_tile_us(kb, nt, f32 != 0); }
extern "C" void deal(const float* cost, const int* tiles, int n, int pairs, unsigned short* out) {
  static uint16_t first[DEAL_CLASSES][DEAL_PAIRS + 1];
  deal_tiles(cost, tiles, n, pairs, first);
  for (int c = 0; c < n; ++c)
    for (int p = 0; p <= pairs; ++p) out[c * (pairs + 1) + p] = first[c][p];
}
""")
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I" + CSRC, str(folder / "d.cpp"), "-o", str(folder / "d.so")], check=True)
    lib = C.CDLL(str(folder / "d.so"))
    lib.tile_us.restype = C.c_float

    def call(cost, tiles, pairs):
        n, out = len(cost), (C.c_ushort * (len(cost) * (pairs + 1)))()
        lib.deal((C.c_float * n)(*cost), (C.c_int * n)(*tiles), n, pairs, out)
        return [list(out[c * (pairs + 1):(c + 1) * (pairs + 1)]) for c in range(n)]
    return call, lib.tile_us


def test_gradient_tiles_are_dealt_out(deal):
    """Every tile to one pair, in order; no pair fuller than the average plus one tile of the costliest class it could lack."""
    call, tile_us = deal
    rng = random.Random(5)
    for _ in range(300):
        n, pairs = rng.randint(1, 6), rng.choice((1, 2, 7, 66, 74, 96))
        cost = sorted((tile_us(rng.randint(1, 200), rng.choice((32, 128, 160, 256)), rng.randint(0, 1)) for _ in range(n)), reverse=True)
        tiles = [rng.choice((1, 3, 28, 74, 75, 672, 9000)) for _ in range(n)]
        first, load, at = call(cost, tiles, pairs), [0.0] * pairs, 0
        for c in range(n):
            assert first[c][0] == at and first[c] == sorted(first[c])
            at += tiles[c]
            assert first[c][pairs] == at
            before = max(load)
            for p in range(pairs):
                load[p] += cost[c] * (first[c][p + 1] - first[c][p])
            assert max(load) <= max(before, sum(load) / pairs + cost[c]) * 1.001 + 1e-3
