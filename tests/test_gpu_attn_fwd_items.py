"""Attention forward with more work items than CTAs: the roles of a CTA walk several items in a row."""
import pytest
import torch

from oracle import attention as A
from test_gpu_parity import attn_inputs, close, f64l, lse_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,S,Hq,Hkv,dh,donor,causal", [
    (13, 104, 12, 12, 64, [0, 0], True),    # one query tile: no item has a second one
    (10, 384, 16, 16, 128, [0], True),      # three: every CTA starts with an item without, some have two in a row
    (6, 264, 15, 3, 64, [0, 0], False),     # the same in full attention, five heads to a KV head
    (13, 104, 12, 6, 64, [0, 0], True),     # an even number of heads to a KV head: two heads' last tiles make an item
    (5, 392, 16, 4, 128, [0, 1], True),
    (4, 257, 20, 10, 64, [0, 0], False),    # one query in the last tile
    (2, 264, 8, 2, 128, [0], True),         # fewer items than SMs: the last tiles stay by themselves
])
def test_items_of_an_odd_number_of_query_tiles(B, S, Hq, Hkv, dh, donor, causal):
    from paper_2608_15943_b200 import kvp
    L = len(donor)
    q, k, v, _ = attn_inputs(B, S, Hq, Hkv, dh, donor)
    o = [torch.full_like(x, float("nan")) for x in q]
    lse = [torch.full((B, Hq, S), float("nan"), device="cuda") for _ in range(L)]
    kvp.attn_fwd(kvp.Shape(L, B, S, 64, Hq, Hkv, dh), donor, q, k, v, o, lse, causal=causal)
    torch.cuda.synchronize()
    assert kvp.device_status() == kvp.OK
    ro, rl = A.attn_fwd(f64l(q), f64l(k), f64l(v), donor, causal=causal)
    for l in range(L):
        close(f"o[{l}]", o[l], ro[l])
        lse_close(f"lse[{l}]", lse[l], rl[l])
