"""Attention forward with more work items than CTAs: the roles of a CTA walk several items in a row."""
import pytest
import torch

from oracle import attention as A
from test_fwd_shape_host import compiled
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


@pytest.fixture(scope="module")
def pack_of(tmp_path_factory):
    return compiled(tmp_path_factory.mktemp("fwd"))


# tiles of 1 << pack heads; the sequence ends in a tile's first token, its last, or between
@pytest.mark.parametrize("B,S,Hq,Hkv,dh,donor,causal,pack", [
    (20, 257, 4, 2, 64, [0], True, 1),       # 64 tokens of two heads: five tiles, the last of one token
    (9, 161, 24, 4, 128, [0], True, 1),      # six heads to a KV head: three groups of two
    (14, 140, 16, 8, 64, [0, 0], False, 1),  # full attention
    (10, 129, 8, 2, 128, [0, 1], True, 2),    # 32 tokens of four heads, the last tile of one token
    (10, 264, 8, 2, 64, [0], True, 2),
    (8, 145, 16, 2, 128, [0, 0], True, 3),   # 16 tokens of eight heads, the last tile of one token
    (4, 272, 24, 3, 64, [0], True, 3),       # every tile full
    (19, 136, 8, 1, 64, [0], False, 3),      # full attention, the last tile half full
    (12, 33, 32, 2, 128, [0, 0], True, 4),   # eight tokens of sixteen heads, five tiles for one key tile
    (5, 136, 32, 2, 64, [0], False, 4),      # every tile full
])
def test_tiles_of_several_heads(pack_of, B, S, Hq, Hkv, dh, donor, causal, pack):
    assert pack_of(B, S, Hq, Hkv, dh, len(donor), int(causal)) == pack
    test_items_of_an_odd_number_of_query_tiles(B, S, Hq, Hkv, dh, donor, causal)


@pytest.mark.parametrize("B,S,Hq,Hkv,dh,pack", [(20, 257, 4, 2, 64, 1), (10, 257, 8, 2, 128, 2), (4, 272, 24, 3, 64, 3)])
def test_fp32_interface_with_tiles_of_several_heads(pack_of, B, S, Hq, Hkv, dh, pack):
    """fp32 tensors that hold bf16 values: the same bits as through the bf16 interface."""
    from paper_2608_15943_b200 import kvp
    assert pack_of(B, S, Hq, Hkv, dh, 1, 1) == pack
    q, k, v, _ = attn_inputs(B, S, Hq, Hkv, dh, [0])
    results = []
    for dtype, code in ((torch.bfloat16, kvp.BF16), (torch.float32, kvp.F32)):
        sh = kvp.Shape(1, B, S, 64, Hq, Hkv, dh, code)
        ws = torch.empty(max(256, kvp.workspace_bytes(kvp.OP_ATTN_FWD, sh, [0])), dtype=torch.uint8, device="cuda")
        o = torch.full(q[0].shape, float("nan"), dtype=dtype, device="cuda")
        lse = torch.full((B, Hq, S), float("nan"), device="cuda")
        kvp.attn_fwd(sh, [0], [q[0].to(dtype)], [k[0].to(dtype)], [v[0].to(dtype)], [o], [lse], ws=ws)
        torch.cuda.synchronize()
        assert kvp.device_status() == kvp.OK
        results.append((o.float(), lse))
    assert torch.equal(results[0][0], results[1][0]) and torch.equal(results[0][1], results[1][1])
