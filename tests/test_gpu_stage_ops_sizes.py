"""RMSNorm, rotary embedding, add and SwiGLU at the edges of how they share the work out: rows per block, heads and pieces
per thread."""
import numpy as np
import pytest
import torch

from oracle import stage as ST
from paper_2608_15943_b200 import synth

pytestmark = pytest.mark.gpu


def bf16_close(got, ref):
    """bf16 storage (half an ulp, at most 2^-8 of the value) of an fp32 computation whose own error is far below."""
    got = got.float().cpu().numpy().astype(np.float64)
    assert np.isfinite(got).all()
    assert (np.abs(got - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-4).all()


@pytest.mark.parametrize("T,D", [(1184, 8), (1185, 2048), (1187, 2056), (2369, 4096), (5, 4104), (1300, 8192)])
def test_rmsnorm_rows_per_block(T, D):
    from paper_2608_15943_b200 import kvp
    x, w = synth.normal((T, D), 61, 1, 1.0, "cuda"), synth.normal((D,), 61, 2, 1.0, "cuda")
    y = torch.full_like(x, float("nan"))
    kvp.rmsnorm(x, w, 1e-5, y)
    bf16_close(y, ST.rmsnorm(x.double().cpu().numpy(), w.double().cpu().numpy(), 1e-5))


@pytest.mark.parametrize("B,S,H,dh,pos0", [(1, 1, 1, 8, 3), (2, 3, 5, 64, 0), (1, 600, 7, 128, 1000), (3, 1200, 9, 256, 0), (1, 9500, 6, 128, 50000)])
def test_rope_heads_per_thread(B, S, H, dh, pos0):
    from paper_2608_15943_b200 import kvp
    x = synth.normal((B, S, H, dh), 62, 1, 1.0, "cuda")
    ref = ST.rope(x.double().cpu().numpy(), 10000.0, pos0)
    bf16_close(kvp.rope(x, 10000.0, pos0), ref)


@pytest.mark.parametrize("n8", [1, 255, 148 * 2048, 148 * 2048 + 1, 2 * 148 * 2048, 2 * 148 * 2048 + 1])
def test_add_and_swiglu_pieces_per_thread(n8):
    """One, two and three 16-byte pieces per thread on a device of 148 SMs, and one more than fits each."""
    from paper_2608_15943_b200 import kvp
    a, b = synth.normal((n8 * 8,), 63, 1, 1.0, "cuda"), synth.normal((n8 * 8,), 63, 2, 1.0, "cuda")
    an, bn = a.double().cpu().numpy(), b.double().cpu().numpy()
    y = torch.full((n8 * 8 + 64,), 7.0, dtype=torch.bfloat16, device="cuda")
    for op, ref in ((kvp.add, an + bn), (kvp.swiglu, ST.swiglu(an, bn))):
        y.fill_(7.0)
        op(a, b, y[:n8 * 8])
        bf16_close(y[:n8 * 8], ref)
        assert (y[n8 * 8:] == 7.0).all()


@pytest.mark.parametrize("T,D", [(1, 4104), (593, 5120), (1777, 6144), (445, 6152), (1333, 8184)])
def test_rmsnorm_wide_rows(T, D):
    """Three and four pieces of a row per thread, one row more than a round of CTAs (four and three per SM)."""
    from paper_2608_15943_b200 import kvp
    x, w = synth.normal((T, D), 64, 1, 1.0, "cuda"), synth.normal((D,), 64, 2, 1.0, "cuda")
    y = torch.full((T + 1, D), 7.0, dtype=torch.bfloat16, device="cuda")
    kvp.rmsnorm(x, w, 1e-5, y[:T])
    bf16_close(y[:T], ST.rmsnorm(x.double().cpu().numpy(), w.double().cpu().numpy(), 1e-5))
    assert (y[T:] == 7.0).all()


@pytest.mark.parametrize("T,D", [(5, 256), (347, 4096), (2400, 1024)])
def test_back_to_back_calls_see_what_the_one_before_wrote(T, D):
    """GEMM, SwiGLU in place, add in place, RMSNorm in place, again and again: the same bits as with a synchronisation after
    every call, although each kernel comes up while the one ahead of it still runs."""
    from paper_2608_15943_b200 import kvp
    w = [synth.normal((D, D), 65, i, 2.0 * D ** -0.5, "cuda") for i in range(2)]
    n = 1.0 + synth.normal((D,), 65, 2, 0.1, "cuda")
    x0 = synth.normal((T, D), 65, 3, 1.0, "cuda")

    def chain(wait):
        x, gate, up = x0.clone(), torch.empty_like(x0), torch.empty_like(x0)
        for _ in range(6):
            for call in (lambda: kvp.gemm(x, w[0], gate), lambda: kvp.gemm(x, w[1], up), lambda: kvp.swiglu(gate, up, gate),
                         lambda: kvp.add(gate, x, x), lambda: kvp.rmsnorm(x, n, 1e-5, x)):
                call()
                if wait:
                    torch.cuda.synchronize()
        torch.cuda.synchronize()
        return x, gate
    want = chain(True)
    assert torch.isfinite(want[0]).all()
    for _ in range(5):
        for got, ref in zip(chain(False), want):
            assert torch.equal(got, ref)


def one_round():
    """16-byte pieces with one for every thread of a full grid of the streaming kernels."""
    return torch.cuda.get_device_properties(0).multi_processor_count * 8 * 256


@pytest.mark.parametrize("rounds,more", [(0, 24), (1, 0), (1, 1), (2, 0), (2, 1), (16, 0), (16, 1)])
def test_swiglu_range_of_gates(rounds, more):
    """Gates over the whole range of exp(-g): overflow, subnormal reciprocals, both infinities (of which the lower has no
    value: -inf / (1 + inf))."""
    from paper_2608_15943_b200 import kvp
    n8 = rounds * one_round() + more
    g, u = synth.normal((n8 * 8,), 66, 1, 8.0, "cuda"), synth.normal((n8 * 8,), 66, 2, 1.0, "cuda")
    special = torch.tensor([0.0, -0.0, 88.0, -86.5, -87.5, -88.0, -88.5, -89.0, -104.0, -3e38, float("inf"), 1e-30, float("-inf")],
                           device="cuda").bfloat16()
    g[:13] = special
    g[-13:] = special
    u[:13] = u[-13:] = 1.0
    y = kvp.swiglu(g, u, torch.full_like(g, 7.0))
    e = torch.exp(-g.double())
    ref = torch.where((e > 3.4028235677973366e38) & (e < float("inf")), -0.0, g.double() / (1.0 + e) * u.double())   # exp(-g) overflows in fp32
    # bf16 storage, and exp(-g) to a few ulps of its argument (|g| 2^-23, at most 2^-16)
    near = (y.double() - ref).abs() <= (2.0 ** -8 + 2.0 ** -15) * ref.abs() + 1e-37
    assert (near | (y.double() == ref) | (y.isnan() & g.isneginf())).all()    # (infinity: equal, but no distance)
    assert y.isnan().sum() == 2


def test_swiglu_does_not_depend_on_the_size():
    """An element's bits are the same in calls of every size: one piece, and either side of one, two and sixteen rounds."""
    from paper_2608_15943_b200 import kvp
    n = (16 * one_round() + 1) * 8
    g, u = synth.normal((n,), 67, 1, 2.0, "cuda"), synth.normal((n,), 67, 2, 1.0, "cuda")
    whole = kvp.swiglu(g, u, torch.full_like(g, float("nan")))
    for n8 in (1, 255, one_round(), one_round() + 1, 2 * one_round(), 2 * one_round() + 1, 16 * one_round()):
        part = kvp.swiglu(g[:n8 * 8], u[:n8 * 8], torch.full((n8 * 8,), float("nan"), dtype=torch.bfloat16, device="cuda"))
        assert torch.equal(part, whole[:n8 * 8]), n8
