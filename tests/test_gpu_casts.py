"""The fp32 interface's conversions of long lists of tensors: more of them than one launch holds."""
import pytest
import torch

from paper_2608_15943_b200 import synth

pytestmark = pytest.mark.gpu


def test_fp32_interface_with_more_tensors_than_one_launch_converts():
    from paper_2608_15943_b200 import kvp
    L, T, D, Hq, Hkv, dh = 23, 12, 64, 2, 1, 64                 # 92 inputs, 69 outputs; 64 per launch
    donor = list(range(L))
    ins = [[synth.normal(s, 41, synth.tid(i, l), 0.2, "cuda") for l in range(L)]
           for i, s in enumerate(((T, D), (Hq * dh, D), (Hkv * dh, D), (Hkv * dh, D)))]
    outs = {}
    for dtype, dt in ((kvp.BF16, torch.bfloat16), (kvp.F32, torch.float32)):
        sh = kvp.Shape(L, 1, T, D, Hq, Hkv, dh, dtype)
        out = [[torch.full((1, T, h, dh), float("nan"), dtype=dt, device="cuda") for _ in range(L)] for h in (Hq, Hkv, Hkv)]
        ws = torch.empty(max(256, kvp.workspace_bytes(kvp.OP_PROJ_FWD, sh, donor)), dtype=torch.uint8, device="cuda")
        kvp.proj_fwd(sh, donor, *([t.to(dt) for t in ts] for ts in ins), *out, ws)
        outs[dt] = [t.float() for ts in out for t in ts]
    for a, b in zip(outs[torch.bfloat16], outs[torch.float32]):
        assert torch.isfinite(a).all() and torch.equal(a, b)


@pytest.mark.parametrize("L,own,S,dh", [(23, 23, 41, 64),    # more tensors than the pre-pass converts beside its own work; three launches
                                        (9, 4, 77, 128),     # two launches, the conversions in the first
                                        (3, 2, 203, 64)])    # two key tiles: accumulators and their conversion too
def test_fp32_attention_backward_is_the_bf16_one(L, own, S, dh):
    """Inputs that are bf16 values: the same dQ, bit for bit up to 128 tokens; the sums up to their order beyond."""
    from paper_2608_15943_b200 import kvp
    B, Hq, Hkv = 2, 4, 2
    donor = [min(l, own - 1) for l in range(L)]
    q, d_o = ([synth.normal((B, S, Hq, dh), 42, synth.tid(i, l), 1.0, "cuda") for l in range(L)] for i in range(2))
    k, v = ([synth.normal((B, S, Hkv, dh), 42, synth.tid(i, l), 1.0, "cuda") if l < own else None for l in range(L)] for i in (2, 3))
    outs = {}
    for dtype, dt in ((kvp.BF16, torch.bfloat16), (kvp.F32, torch.float32)):
        sh = kvp.Shape(L, B, S, 64, Hq, Hkv, dh, dtype)
        tq, tk, tv, td = ([None if t is None else t.to(dt) for t in ts] for ts in (q, k, v, d_o))
        o, lse = [torch.empty_like(t) for t in tq], [torch.empty(B, Hq, S, device="cuda") for _ in range(L)]
        dq = [torch.full_like(t, float("nan")) for t in tq]
        dk, dv = ([None if t is None else torch.full(t.shape, float("nan"), device="cuda") for t in k] for _ in range(2))
        ws = torch.empty(max(256, *(kvp.workspace_bytes(op, sh, donor) for op in (kvp.OP_ATTN_FWD, kvp.OP_ATTN_BWD))), dtype=torch.uint8, device="cuda")
        kvp.attn_fwd(sh, donor, tq, tk, tv, o, lse, ws=ws)
        kvp.attn_bwd(sh, donor, tq, tk, tv, o, td, lse, dq, dk, dv, ws)
        assert kvp.device_status() == kvp.OK
        outs[dt] = [t.float() for t in dq + dk + dv if t is not None]
    for a, b in zip(outs[torch.bfloat16], outs[torch.float32]):
        assert torch.isfinite(a).all()
        # beyond one key tile two partials a dQ element and a few per dK / dV element, in any order: half an ulp of bf16 at most
        # where the rounded sums differ, and that rarely
        assert torch.equal(a, b) if S <= 128 else (a - b).norm() <= 1e-3 * a.norm()
