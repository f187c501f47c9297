"""Decode when the library deals the K/V rows out: shares that begin and end anywhere in the list of all sequences."""
import numpy as np
import pytest
import torch

from oracle import attention as A
from test_gpu_parity import ABS, LSE_TOL, REL, f64, f64l
from paper_2608_15943_b200 import synth

pytestmark = pytest.mark.gpu


def dense(pool, bt, lens, page):
    """[B, cap, Hkv, dh] from the pages of each sequence."""
    out = np.zeros((len(lens), max(lens), pool.shape[1], pool.shape[3]))
    for b, n in enumerate(lens):
        rows = pool[bt[b, :(n + page - 1) // page].long()].permute(0, 2, 1, 3).reshape(-1, pool.shape[1], pool.shape[3])
        out[b, :n] = f64(rows[:n])
    return out


@pytest.mark.parametrize("L,donor,B,Hq,Hkv,dh,page,lens,static", [
    (1, [0], 1, 1, 1, 128, 16, [1], False),                              # one granule, one block
    (1, [0], 1, 4, 1, 128, 128, [20000], False),                         # one unit over many blocks: eight warps a row in the merge
    (1, [0], 1, 16, 1, 64, 64, [9001], False),                           # the same at dh 64, all 16 rows
    (2, [0, 0], 40, 8, 2, 128, 16, [17 + 13 * b for b in range(40)], False),   # more than 32 lengths; units of 2 to 34 granules
    (3, [0, 1, 2], 33, 2, 2, 64, 32, [16] * 33, False),                  # units of one granule, dealt out whole
    (2, [0, 1], 3, 4, 4, 128, 16, [1100, 3, 900], False),                # units of 1 to 69 granules, two groups
    (4, [0, 0, 0, 0], 3, 12, 2, 128, 32, [640, 1, 333], True),           # 16-row passes of uneven groups; built-in scratch
])
def test_decode_shares(L, donor, B, Hq, Hkv, dh, page, lens, static):
    from paper_2608_15943_b200 import kvp
    max_pages = (max(lens) + page - 1) // page + 1
    n_pages = sum((n + page - 1) // page for n in lens)
    order = torch.randperm(n_pages, generator=torch.Generator().manual_seed(9)).int()
    bt, at = torch.zeros(B, max_pages, dtype=torch.int32), 0
    for b, n in enumerate(lens):
        k = (n + page - 1) // page
        bt[b, :k] = order[at:at + k]
        at += k
    own = [l for l in range(L) if donor[l] == l]
    mk = lambda kind: [synth.normal((n_pages, Hkv, page, dh), 51, synth.tid(kind, l), 1.0, "cuda") if l in own else None for l in range(L)]
    kc, vc = mk(7), mk(8)
    for b, n in enumerate(lens):                                         # slots never appended hold NaN
        if n % page:
            for l in own:
                kc[l][bt[b, n // page].long(), :, n % page:] = float("nan")
                vc[l][bt[b, n // page].long(), :, n % page:] = float("nan")
    q = [synth.normal((B, Hq, dh), 51, synth.tid(6, l), 1.0, "cuda") for l in range(L)]
    o = [torch.full((B, Hq, dh), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(L)]
    lse = [torch.full((B, Hq), float("nan"), device="cuda") for _ in range(L)]
    desc = kvp.DecodeDesc(L, B, Hq, Hkv, dh, page, max_pages, n_pages)
    lengths = torch.tensor(lens, dtype=torch.int32, device="cuda")
    if static:
        kvp.decode_static(desc, donor, q, kc, vc, bt.cuda(), lengths, o, lse)
    else:
        ws = torch.empty(kvp.decode_workspace_bytes(desc, donor), dtype=torch.uint8, device="cuda")
        kvp.decode(desc, donor, q, kc, vc, bt.cuda(), lengths, o, lse, ws)
    torch.cuda.synchronize()
    assert kvp.device_status() == kvp.OK
    kd = [dense(kc[l], bt, lens, page) if l in own else None for l in range(L)]
    vd = [dense(vc[l], bt, lens, page) if l in own else None for l in range(L)]
    ro, rl = A.decode_attend(f64l(q), kd, vd, lens, donor)
    for l in range(L):
        got = f64(o[l])
        assert np.isfinite(got).all()
        assert np.linalg.norm(got - ro[l]) <= REL * np.linalg.norm(ro[l])
        assert np.abs(got - ro[l]).max() <= ABS
        assert np.abs(f64(lse[l]) - rl[l]).max() <= LSE_TOL
