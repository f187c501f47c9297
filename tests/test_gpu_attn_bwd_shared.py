"""Attention backward with gradients in the memory of inputs."""
import pytest
import torch

from paper_2608_15943_b200 import synth

pytestmark = pytest.mark.gpu


def inputs(B, S, Hq, Hkv, dh, donor, dt):
    """q, k, v, o, lse, d_o of the layers, from the forward pass."""
    from paper_2608_15943_b200 import kvp
    L = len(donor)
    q, d_o = ([synth.normal((B, S, Hq, dh), 43, synth.tid(i, l), 1.0, "cuda").to(dt) for l in range(L)] for i in range(2))
    k, v = ([synth.normal((B, S, Hkv, dh), 43, synth.tid(i, l), 1.0, "cuda").to(dt) if donor[l] == l else None for l in range(L)] for i in (2, 3))
    sh = kvp.Shape(L, B, S, 64, Hq, Hkv, dh, kvp.F32 if dt == torch.float32 else kvp.BF16)
    o, lse = [torch.empty_like(t) for t in q], [torch.empty(B, Hq, S, device="cuda") for _ in range(L)]
    ws = torch.empty(max(256, *(kvp.workspace_bytes(op, sh, donor) for op in (kvp.OP_ATTN_FWD, kvp.OP_ATTN_BWD))), dtype=torch.uint8, device="cuda")
    kvp.attn_fwd(sh, donor, q, k, v, o, lse, ws=ws)
    return dict(q=q, k=k, v=v, o=o, d_o=d_o, lse=lse), sh, ws


def backward(ins, sh, ws, donor, place):
    """Gradients as fp32; place(name, layer, copies of the inputs): the tensor a gradient is written to, or None."""
    from paper_2608_15943_b200 import kvp
    t = {n: [None if x is None else x.clone() for x in xs] for n, xs in ins.items()}
    fresh = lambda like, dt: torch.full(like.shape, float("nan"), dtype=dt, device="cuda")

    def out(name, l, like, dt):
        p = place(name, l, t)
        return fresh(like, dt) if p is None else p
    dq = [out("dq", l, x, x.dtype) for l, x in enumerate(t["q"])]
    dk, dv = ([out(n, l, x, torch.float32) if x is not None else None for l, x in enumerate(t["k"])] for n in ("dk", "dv"))
    kvp.attn_bwd(sh, donor, t["q"], t["k"], t["v"], t["o"], t["d_o"], t["lse"], dq, dk, dv, ws)
    torch.cuda.synchronize()
    assert kvp.device_status() == kvp.OK
    return [x.float() for x in dq + dk + dv if x is not None]


def same(a, b, S):
    for x, y in zip(a, b):
        assert torch.isfinite(x).all()
        # up to 128 tokens the same bits; beyond, sums of a few fp32 terms in any order, rounded to bf16 in dq: half an ulp where
        # the rounded sums differ, and that rarely
        assert torch.equal(x, y) if S <= 128 else (x - y).norm() <= 1e-3 * x.norm()


IN_PLACE = {
    "dk over k, dv over v, dq over q": lambda n, l, t: t[{"dk": "k", "dv": "v", "dq": "q"}[n]][l],
    "dk over dO, dv over O": lambda n, l, t: t[{"dk": "d_o", "dv": "o"}[n]][l] if n != "dq" else None,
    "dq over O and dO of layers of another launch": lambda n, l, t: t["o" if l % 2 else "d_o"][-1 - l] if n == "dq" else None,
    "dv over q of the last layer": lambda n, l, t: t["q"][-1] if (n, l) == ("dv", 0) else None,
}


@pytest.mark.parametrize("case", IN_PLACE)
@pytest.mark.parametrize("B,S,H,dh,L", [(2, 96, 4, 64, 3), (1, 300, 2, 128, 2), (1, 72, 2, 64, 18), (1, 40, 2, 64, 23)])   # one launch; several; more tensors than a pre-pass rounds
def test_fp32_gradients_in_place_of_inputs(case, B, S, H, dh, L):
    """The inputs are read, all of them, before a gradient is written."""
    donor = list(range(L))
    ins, sh, ws = inputs(B, S, H, H, dh, donor, torch.float32)
    want = backward(ins, sh, ws, donor, lambda n, l, t: None)
    same(want, backward(ins, sh, ws, donor, IN_PLACE[case]), S)


DQ_OVER = {   # up to 128 tokens the kernel that reads q, k, v and d_o writes dQ too, where it has read what lies there
    "q": lambda l, t: t["q"][l],
    "d_o": lambda l, t: t["d_o"][l],
    "o": lambda l, t: t["o"][l],
    "k or v": lambda l, t: t["kv"[l % 2]][l],
    "q of another layer": lambda l, t: t["q"][-1 - l],
    "d_o of another layer": lambda l, t: t["d_o"][l - 1],
}


@pytest.mark.parametrize("over", DQ_OVER)
@pytest.mark.parametrize("B,S,H,dh,L", [(2, 128, 4, 64, 4), (3, 41, 2, 128, 3), (1, 65, 8, 128, 8), (1, 200, 2, 64, 2)])
def test_dq_in_place_of_inputs(over, B, S, H, dh, L):
    donor = list(range(L))
    ins, sh, ws = inputs(B, S, H, H, dh, donor, torch.bfloat16)
    want = backward(ins, sh, ws, donor, lambda n, l, t: None)
    same(want, backward(ins, sh, ws, donor, lambda n, l, t: DQ_OVER[over](l, t) if n == "dq" else None), S)
