"""Backward CTAs that take part of the query streams of a small window (short sequences, few of them)."""
import pytest
import torch

from oracle import attention as A
from test_gpu_parity import attn_inputs, close, f64l

pytestmark = pytest.mark.gpu


def backward(kvp, B, S, Hq, Hkv, dh, donor, causal, inputs):
    L = len(donor)
    q, k, v, d_o = inputs
    sh = kvp.Shape(L, B, S, 64, Hq, Hkv, dh)
    o, lse = [torch.empty_like(x) for x in q], [torch.empty(B, Hq, S, device="cuda") for _ in range(L)]
    kvp.attn_fwd(sh, donor, q, k, v, o, lse, causal=causal)
    dq = [torch.full_like(x, float("nan")) for x in q]
    dk, dv = ([torch.full((B, S, Hkv, dh), float("nan"), device="cuda") if d == l else None for l, d in enumerate(donor)] for _ in range(2))
    ws = torch.empty(kvp.workspace_bytes(kvp.OP_ATTN_BWD, sh, donor), dtype=torch.uint8, device="cuda")
    kvp.attn_bwd(sh, donor, q, k, v, o, d_o, lse, dq, dk, dv, ws, causal=causal)
    torch.cuda.synchronize()
    assert kvp.device_status() == kvp.OK
    return dq, dk, dv


@pytest.mark.parametrize("B,S,Hq,Hkv,dh,donor,causal", [
    (1, 64, 12, 2, 128, [0, 0], True),             # one query tile: the streams in two parts
    (2, 128, 8, 1, 64, [0, 0, 0], True),           # two windows of one query tile
    (1, 161, 16, 1, 128, [0, 0, 0, 0, 0], False),  # 80 streams over one- and two-tile windows, parts of unequal size
    (1, 321, 7, 1, 64, [0, 1, 1], True),           # an odd number of streams, rows past the end in the last 32-row slice
])
def test_backward_in_parts(B, S, Hq, Hkv, dh, donor, causal):
    from paper_2608_15943_b200 import kvp
    inputs = attn_inputs(B, S, Hq, Hkv, dh, donor)
    dq, dk, dv = backward(kvp, B, S, Hq, Hkv, dh, donor, causal, inputs)
    rq, rk, rv = A.attn_bwd(*(f64l(x) for x in inputs), donor, causal=causal)
    for l, d in enumerate(donor):
        close(f"dq[{l}]", dq[l], rq[l])
        if d == l:
            close(f"dk[{l}]", dk[l], rk[l], sum_over_tokens=True)
            close(f"dv[{l}]", dv[l], rv[l], sum_over_tokens=True)
    if S <= 128:                                   # one key tile: the same bits in every run
        again = backward(kvp, B, S, Hq, Hkv, dh, donor, causal, inputs)
        for a, b in zip(dq + dk + dv, again[0] + again[1] + again[2]):
            assert (a is None and b is None) or torch.equal(a, b)


@pytest.mark.parametrize("dh", [64, 128])
@pytest.mark.parametrize("S", [9, 47, 79, 321])   # ends inside an eight, a sixteen and a tile of queries; more steps than any ring holds
def test_dq_of_ragged_tiles(S, dh):
    from paper_2608_15943_b200 import kvp
    inputs = attn_inputs(2, S, 6, 2, dh, [0, 0])
    dq = backward(kvp, 2, S, 6, 2, dh, [0, 0], True, inputs)[0]
    rq = A.attn_bwd(*(f64l(x) for x in inputs), [0, 0], causal=True)[0]
    for l in range(2):
        close(f"dq[{l}]", dq[l], rq[l])
