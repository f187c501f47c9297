"""RMSNorm and rotary embedding at the edges of how they share the work out: one row or two per block, all heads or a
few per thread."""
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
