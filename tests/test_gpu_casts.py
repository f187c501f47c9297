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
