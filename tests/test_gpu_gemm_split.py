"""GEMMs with few rows of A (decode-step projections, prompts): operands swapped, K split over a cluster of CTAs, or tiles
of tokens on CTA pairs; and the weight and input gradients, which take those pairs too."""
import pytest
import torch

from guard import Guarded
from paper_2608_15943_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [
    (1, 8, 8),            # less than one tile and one k-block: split 1
    (16, 128, 64), (17, 136, 72),          # edges of the token tile, the column tile and the k-block
    (31, 264, 1032),      # split 8, 17 k-blocks dealt unevenly
    (128, 4096, 520),     # widest token tile; 32 column tiles: split 4
    (40, 19208, 200),     # more CTAs than SMs: two per SM, shallow ring, split 1
    (129, 4104, 2056),    # first row count of the chosen kernels: K split, one ragged column tile
    (347, 520, 2048),     # K split in four, several token tiles, the last one short
    (200, 11016, 136),    # CTA pairs with one short token tile
    (513, 5512, 1032),    # three token tiles of 192, the last of 129, 22 column tiles
    (289, 16392, 136),    # more tiles than pairs, the last column tile of eight columns
    (2049, 2056, 200),    # thirteen token tiles of 160, nine column tiles
    (1300, 8200, 72),     # several rounds of tiles, pairs in alternating direction
])
def test_few_rows(M, N, K):
    from paper_2608_15943_b200 import kvp
    a = synth.normal((M, K), 31, 1, 1.0, "cuda")
    b = synth.normal((N, K), 31, 2, 1.0, "cuda")
    ref = a.double() @ b.double().T
    gd = Guarded()
    c32 = gd.empty((M, N), torch.float32, float("nan"))
    c16 = gd.empty((M, N), torch.bfloat16, float("nan"))
    kvp.gemm(a, b, c32)
    kvp.gemm(a, b, c16)
    gd.check()
    assert kvp.device_status() == kvp.OK
    # fp32 accumulation of K products of bf16 values (each product exact): |error| <= K 2^-24 sum|a b|, of which the
    # average case is far below; bf16 storage (8 significant bits) adds half an ulp, at most 2^-8 of the value
    bound = K * 2.0 ** -24 * (a.double().abs() @ b.double().abs().T) + 1e-30
    assert ((c32.double() - ref).abs() <= bound).all()
    assert ((c16.double() - ref).abs() <= bound + 2.0 ** -8 * ref.abs()).all()


@pytest.mark.parametrize("M,N,K", [(5, 4104, 4104), (128, 11016, 1608), (33, 18440, 920), (70, 1032, 16400)])
def test_few_rows_streamed_b(M, N, K):
    """B just above a quarter of L2, read with a cache policy: two accumulators, one, no split, eight pieces of K."""
    test_few_rows(M, N, K)


def test_few_rows_grouped_projections():
    """Q, K and V projections of twelve layers with one token per sequence: 20 problems in one launch, two widths."""
    from paper_2608_15943_b200 import kvp
    L, B, D, Hq, Hkv, dh = 12, 5, 256, 4, 2, 64
    donor = [0, 1, 2, 3, 3, 3, 3, 3, 3, 3, 3, 3]
    sh = kvp.Shape(L, B, 1, D, Hq, Hkv, dh)
    x = [synth.normal((B, D), 32, synth.tid(0, l), 1.0, "cuda") for l in range(L)]
    w = {n: [synth.normal((h * dh, D), 32, synth.tid(i, l), 0.02, "cuda") for l in range(L)]
         for i, (n, h) in enumerate((("q", Hq), ("k", Hkv), ("v", Hkv)), 1)}
    gd = Guarded()
    out = {n: [gd.empty((B, 1, h, dh), torch.bfloat16, float("nan")) for _ in range(L)] for n, h in (("q", Hq), ("k", Hkv), ("v", Hkv))}
    kvp.proj_fwd(sh, donor, x, w["q"], w["k"], w["v"], out["q"], out["k"], out["v"])
    gd.check()
    for l in range(L):
        for n in ("q", "k", "v") if donor[l] == l else ("q",):
            ref = x[l].double() @ w[n][l].double().T
            got = out[n][l].view(B, -1).double()
            assert ((got - ref).abs() <= 2.0 ** -8 * ref.abs() + 1e-4).all(), (n, l)   # bf16 storage; 256 terms of size 0.02


@pytest.mark.parametrize("L,own,S,D,Hq,Hkv", [
    (1, 1, 8, 64, 1, 1),          # the fewest tokens: less than one k-block along them, eight rows of dX
    (4, 1, 136, 320, 2, 1),       # tiles of 128 rows, remainders rounded up to 32 (dX) and to 128 (MN-major A)
    (5, 2, 392, 1088, 6, 3),      # tiles of 256 rows, one and three K segments
    (20, 8, 104, 576, 4, 1),       # more problems than one launch holds
    (1, 1, 7048, 4096, 64, 16),   # above the line to single-CTA tiles
    (6, 5, 264, 1088, 66, 6),     # tiles dealt out by cost, two equal ones along the tokens; eight epilogue warps a tile
    (2, 1, 296, 2112, 20, 2),     # dealt out, all epilogue warps on every tile
])
def test_gradient_gemms(L, own, S, D, Hq, Hkv):
    from paper_2608_15943_b200 import kvp
    dh, T = 64, S
    donor = [min(l, own - 1) for l in range(L)]
    sh = kvp.Shape(L, 1, S, D, Hq, Hkv, dh)
    x = [synth.normal((T, D), 33, synth.tid(0, l), 1.0, "cuda") for l in range(L)]
    w = {n: [synth.normal((h * dh, D), 33, synth.tid(i, l), 0.5, "cuda") for l in range(L)]
         for i, (n, h) in enumerate((("q", Hq), ("k", Hkv), ("v", Hkv)), 1)}
    dq = [synth.normal((T, Hq * dh), 33, synth.tid(4, l), 1.0, "cuda") for l in range(L)]
    dkv = [[synth.normal((T, Hkv * dh), 33, synth.tid(i, l), 1.0, "cuda").float() if l < own else None for l in range(L)] for i in (5, 6)]
    ws = torch.empty(kvp.workspace_bytes(kvp.OP_PROJ_BWD, sh, donor), dtype=torch.uint8, device="cuda")
    gd = Guarded()
    dw = {n: [gd.empty((h * dh, D), torch.float32, float("nan")) if n == "q" or l < own else None for l in range(L)]
          for n, h in (("q", Hq), ("k", Hkv), ("v", Hkv))}
    dx = [gd.empty((T, D), torch.bfloat16, float("nan")) for _ in range(L)]
    kvp.proj_bwd(sh, donor, x, w["q"], w["k"], w["v"], dq, dkv[0], dkv[1], dw["q"], dw["k"], dw["v"], dx, ws)
    gd.check()
    assert kvp.device_status() == kvp.OK
    for l in range(L):
        parts = [("q", dq[l])] + ([("k", dkv[0][l]), ("v", dkv[1][l])] if l < own else [])
        # as test_few_rows: K 2^-24 sum|a b| for the fp32 sums, half an ulp of bf16 for dX
        for n, d in parts:
            bound = T * 2.0 ** -24 * (d.double().abs().T @ x[l].double().abs()) + 1e-30
            assert ((dw[n][l].double() - d.double().T @ x[l].double()).abs() <= bound).all(), (n, l)
        ref = sum(d.double() @ w[n][l].double() for n, d in parts)
        K = sum(d.shape[1] for _, d in parts)
        bound = K * 2.0 ** -24 * sum(d.double().abs() @ w[n][l].double().abs() for n, d in parts)
        assert ((dx[l].double() - ref).abs() <= bound + 2.0 ** -8 * ref.abs()).all(), l


@pytest.mark.parametrize("L", [1, 2, 3, 4, 5, 8, 9])      # L problems forward, 2 L backward: parameter blocks of 1, 4, 8 and 32
@pytest.mark.parametrize("T,kind", [(40, "split"), (200, "tall")])
def test_parameter_blocks_of_each_size(choose, L, T, kind):
    from paper_2608_15943_b200 import kvp
    D, Hq, dh = 1024, 1, 64
    N = Hq * dh
    assert ("single", "pair", "tall", "split")[choose([(T, D, N)] * L)[0]] == kind
    sh = kvp.Shape(L, 1, T, D, Hq, 1, dh)
    o, wo, dy = ([synth.normal(s, 37, synth.tid(i, l), 1.0, "cuda") for l in range(L)] for i, s in enumerate(((T, N), (D, N), (T, D))))
    gd = Guarded()
    y, d_o = ([gd.empty(s, torch.bfloat16, float("nan")) for _ in range(L)] for s in ((T, D), (T, N)))
    dwo = [gd.empty((D, N), torch.float32, float("nan")) for _ in range(L)]
    kvp.out_proj_fwd(sh, o, wo, y)
    kvp.out_proj_bwd(sh, o, wo, dy, d_o, dwo)
    gd.check()
    assert kvp.device_status() == kvp.OK
    for l in range(L):
        for got, a, b in ((y[l], o[l], wo[l].T), (d_o[l], dy[l], wo[l]), (dwo[l], dy[l].T, o[l])):
            a, b = a.double(), b.double()
            half_ulp = 2.0 ** -8 * (a @ b).abs() if got.dtype == torch.bfloat16 else 0.0      # bounds as test_few_rows
            assert ((got.double() - a @ b).abs() <= a.shape[1] * 2.0 ** -24 * (a.abs() @ b.abs()) + half_ulp + 1e-30).all()


@pytest.fixture(scope="module")
def choose(tmp_path_factory):
    from test_gemm_choice_host import compiled
    return compiled(tmp_path_factory.mktemp("choice"))[0]


@pytest.fixture(scope="module")
def split_choice(tmp_path_factory):
    from test_gemm_choice_host import compiled
    return compiled(tmp_path_factory.mktemp("split"))[1]


# (kernel, tokens per tile, K split) that a launch is to take: a change of the rules that moves a case off the edge it is
# here for fails instead of passing somewhere else
@pytest.mark.parametrize("M,N,K,kernel", [
    (193, 264, 8, ("tall", 96, 1)), (207, 264, 8, ("tall", 96, 1)), (209, 1032, 8, ("tall", 96, 1)),    # last tiles of 1, 15, 17 tokens
    (1345, 9688, 136, ("tall", 224, 1)), (1360, 9688, 136, ("tall", 224, 1)), (1375, 9688, 136, ("tall", 224, 1)),   # 1, 16, 31; 38 columns of 7 tiles
    (961, 5512, 200, ("tall", 192, 1)), (1280, 9688, 136, ("tall", 256, 1)),                             # the largest tile, no remainder
    (145, 264, 2056, ("split", 48, 4)), (159, 520, 1032, ("split", 48, 4)), (401, 520, 1032, ("split", 48, 2)), (192, 1032, 520, ("split", 48, 1)),
    (279, 9688, 8, ("single", 0, 1)), (290, 9608, 16, ("single", 0, 1)),                                # single-CTA tiles, last of 23 and 34 rows
    (3897, 19016, 8, ("pair", 0, 1)),                                                                   # CTA pairs, last rows 57, last columns 72
    (4097, 520, 72, ("pair", 0, 1)), (4224, 264, 136, ("pair", 0, 1)),                                  # the first row counts without a choice
])
def test_each_forward_kernel_at_its_edges(choose, M, N, K, kernel):
    from paper_2608_15943_b200 import kvp
    kind, nt, split = choose([(M, N, K)])
    assert (("single", "pair", "tall", "split")[kind], nt, split) == kernel
    test_few_rows(M, N, K)


# tokens per tile, CTAs of a cluster and accumulators of a CTA in the kernel of few rows: short last tiles of tokens, columns
# and k-blocks, both sides of the line from which a warp sums several tokens at a time (more than twelve per CTA of clusters
# of one and two), the longest tile with every cluster, rings of three stages (more CTAs than SMs)
@pytest.mark.parametrize("M,N,K,nt,split,parts", [
    (16, 136, 1032, 16, 8, 1), (16, 8200, 520, 16, 2, 1), (33, 8200, 520, 48, 2, 1), (30, 2056, 2056, 32, 4, 2), (33, 136, 1032, 32, 8, 1),
    (33, 1032, 1032, 48, 8, 1), (70, 5512, 2056, 80, 4, 1), (97, 4104, 4104, 112, 4, 1), (128, 2056, 2056, 128, 4, 2),
    (128, 2048, 2056, 64, 4, 2), (113, 4616, 648, 64, 2, 2), (17, 4616, 4104, 16, 2, 2), (9, 4616, 200, 16, 2, 2),
    (127, 8, 8, 32, 1, 1), (65, 264, 72, 48, 2, 1), (113, 520, 136, 32, 2, 1), (97, 648, 200, 32, 4, 1), (65, 520, 520, 48, 8, 1),
    (128, 17416, 72, 128, 1, 1), (113, 19208, 200, 128, 1, 1), (115, 8200, 4104, 128, 2, 1), (128, 11016, 136, 128, 2, 1),
    (128, 4104, 8200, 128, 4, 1), (113, 5512, 520, 128, 4, 1), (115, 1544, 648, 128, 8, 1), (113, 2824, 520, 128, 8, 1),
])
def test_few_rows_sums(split_choice, M, N, K, nt, split, parts):
    assert split_choice([(M, N, K)])[:3] == (nt, split, parts)
    test_few_rows(M, N, K)


@pytest.mark.parametrize("N,K", [(8, 72), (136, 1032), (520, 520), (1544, 648), (2056, 2056), (2824, 8200), (5512, 4104), (11016, 136), (19208, 200)])
def test_a_row_does_not_depend_on_the_number_of_rows(N, K):
    """Up to 128 rows the pieces of K, with an accumulator each, go by the columns and the depth: a row has the same bits
    whichever tiles and clusters the call takes.  """
    from paper_2608_15943_b200 import kvp
    a, b = synth.normal((128, K), 35, 1, 1.0, "cuda"), synth.normal((N, K), 35, 2, 1.0, "cuda")
    whole = kvp.gemm(a, b, torch.full((128, N), float("nan"), device="cuda"))
    for M in (1, 16, 17, 33, 64, 65, 100, 127):
        few = kvp.gemm(a[:M], b, torch.full((M, N), float("nan"), device="cuda"))
        assert torch.equal(few, whole[:M]), M
    assert kvp.device_status() == kvp.OK


# three problems of one launch, and six, of more than 96 rows
@pytest.mark.parametrize("owners,D,Hq,Hkv,nt,split,parts", [
    (1, 576, 2, 1, 32, 8, 1), (1, 1536, 24, 4, 64, 4, 2), (1, 2048, 32, 8, 128, 8, 1), (2, 1536, 8, 4, 64, 4, 2), (2, 192, 24, 8, 128, 2, 1),
    (2, 576, 48, 8, 128, 2, 1),
])
def test_many_rows_of_grouped_projections(split_choice, owners, D, Hq, Hkv, nt, split, parts):
    from paper_2608_15943_b200 import kvp
    B, dh = 113, 64
    assert split_choice([(B, Hq * dh, D), (B, Hkv * dh, D), (B, Hkv * dh, D)] * owners)[:3] == (nt, split, parts)
    sh = kvp.Shape(owners, B, 1, D, Hq, Hkv, dh)
    x = [synth.normal((B, D), 36, synth.tid(0, l), 1.0, "cuda") for l in range(owners)]
    w = {n: [synth.normal((h * dh, D), 36, synth.tid(i, l), 1.0, "cuda") for l in range(owners)]
         for i, (n, h) in enumerate((("q", Hq), ("k", Hkv), ("v", Hkv)), 1)}
    gd = Guarded()
    out = {n: [gd.empty((B, 1, h, dh), torch.bfloat16, float("nan")) for _ in range(owners)] for n, h in (("q", Hq), ("k", Hkv), ("v", Hkv))}
    kvp.proj_fwd(sh, list(range(owners)), x, w["q"], w["k"], w["v"], out["q"], out["k"], out["v"])
    gd.check()
    assert kvp.device_status() == kvp.OK
    for l in range(owners):
        for n in ("q", "k", "v"):
            ref = x[l].double() @ w[n][l].double().T
            bound = D * 2.0 ** -24 * (x[l].double().abs() @ w[n][l].double().abs().T)     # as test_few_rows
            assert ((out[n][l].view(B, -1).double() - ref).abs() <= bound + 2.0 ** -8 * ref.abs()).all(), (n, l)


@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("M,N,K,cols", [(129, 8, 72, 24), (160, 264, 136, 520), (300, 520, 64, 528), (513, 296, 200, 304)])
def test_results_inside_a_wider_matrix(mode, M, N, K, cols):
    """C is a block of columns of a wider matrix: the tile kernels store whole boxes of it, and nothing beside it."""
    from paper_2608_15943_b200 import kvp
    a, b = synth.normal((M, K), 34, 1, 1.0, "cuda"), synth.normal((N, K), 34, 2, 1.0, "cuda")
    ref = a.double() @ b.double().T
    bound = K * 2.0 ** -24 * (a.double().abs() @ b.double().abs().T) + 1e-30   # as test_few_rows
    kvp.set_gemm_pair_mode(mode)
    try:
        for dtype in (torch.bfloat16, torch.float32):
            whole = torch.full((M + 3, cols), 7.0, dtype=dtype, device="cuda")
            c = whole[1:M + 1, 8:8 + N]
            kvp.gemm(a, b, c)
            assert kvp.device_status() == kvp.OK
            half_ulp = 2.0 ** -8 * ref.abs() if dtype == torch.bfloat16 else 0.0
            assert ((c.double() - ref).abs() <= bound + half_ulp).all()
            c.fill_(7.0)
            assert (whole == 7.0).all()
    finally:
        kvp.set_gemm_pair_mode(1)
