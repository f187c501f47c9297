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


def paged(lens, Hkv, dh, page, seed):
    """Pools of one layer with the pages of each sequence in a row, their block table and max_pages."""
    need = [(n + page - 1) // page for n in lens]
    bt, at = torch.zeros(len(lens), max(need), dtype=torch.int32), 0
    for b, k in enumerate(need):
        bt[b, :k] = torch.arange(at, at + k)
        at += k
    return [synth.normal((at, Hkv, page, dh), seed, i, 1.0, "cuda") for i in (1, 2)] + [bt]


def exact_on_gpu(q, kc, vc, bt, lens, page):
    """The oracle's decode in 64 bits for sizes that take numpy too long: outputs [B, Hq, dh] and LSE [B, Hq]."""
    B, Hq, dh = q.shape
    Hkv = kc.shape[1]
    o, lse = torch.empty(B, Hq, dh, dtype=torch.float64, device="cuda"), torch.empty(B, Hq, dtype=torch.float64, device="cuda")
    for b, n in enumerate(lens):
        k, v = (p[bt[b, :(n + page - 1) // page].long().cuda()].permute(1, 0, 2, 3).reshape(Hkv, -1, dh)[:, :n].double() for p in (kc, vc))
        s = torch.einsum("hgd,hnd->hgn", q[b].double().view(Hkv, Hq // Hkv, dh), k) * dh ** -0.5
        o[b] = torch.einsum("hgn,hnd->hgd", torch.softmax(s, -1), v).reshape(Hq, dh)
        lse[b] = torch.logsumexp(s, -1).reshape(Hq)
    return o, lse


def decode_one_layer(q, kc, vc, bt, lens, page, num_splits=0):
    from paper_2608_15943_b200 import kvp
    B, Hq, dh = q.shape
    desc = kvp.DecodeDesc(1, B, Hq, kc.shape[1], dh, page, bt.shape[1], kc.shape[0], num_splits)
    o, lse = torch.full_like(q, float("nan")), torch.full((B, Hq), float("nan"), device="cuda")
    ws = torch.empty(kvp.decode_workspace_bytes(desc, [0]), dtype=torch.uint8, device="cuda")
    kvp.decode(desc, [0], [q], [kc], [vc], bt.cuda(), torch.tensor(lens, dtype=torch.int32, device="cuda"), [o], [lse], ws)
    assert kvp.device_status() == kvp.OK
    return o.double(), lse.double()


def test_error_does_not_grow_with_the_share():
    """Shares of 166 granules are no further from 64 bits than splits of 128 (2048 tokens): a warp's 41 granules against 32.
    With 32768 outputs two draws of the same error differ by 0.4 % (one sigma); 1 % is allowed."""
    lens, page = [16384] * 8, 128
    kc, vc, bt = paged(lens, 8, 128, page, 71)
    q = synth.normal((8, 32, 128), 71, 3, 1.0, "cuda")
    ro, rl = exact_on_gpu(q, kc, vc, bt, lens, page)
    got, lse = decode_one_layer(q, kc, vc, bt, lens, page)
    split, _ = decode_one_layer(q, kc, vc, bt, lens, page, num_splits=8)
    assert (got - ro).norm() <= 1.01 * (split - ro).norm()
    assert (lse - rl).abs().max() <= 2e-6     # values of about 10: two ulps


@pytest.mark.parametrize("at", [0, 700, 4999])
def test_one_score_far_above_the_others(at):
    """One token 290 (log2) above the rest, first, in the middle or last: what comes before it vanishes and what comes after
    it adds nothing, however often the reference of the probabilities falls."""
    lens, page = [5000], 16
    kc, vc, bt = paged(lens, 1, 64, page, 72)
    q = synth.normal((1, 4, 64), 72, 3, 1.0, "cuda")
    q[:, 1:] = q[:, :1]
    kc[at // page, 0, at % page] = q[0, 0] * 25.0
    ro, rl = exact_on_gpu(q, kc, vc, bt, lens, page)
    got, lse = decode_one_layer(q, kc, vc, bt, lens, page)
    assert (got - ro).norm() <= REL * ro.norm() and (lse - rl).abs().max() <= 2e-7 * rl.abs().max()


@pytest.mark.parametrize("lens,Hkv,dh,page", [
    ([32768] + [300] * 63, 8, 128, 128),                  # short units on average, one of 2048 granules
    ([200] * 20 + [30000] + [200] * 19, 4, 64, 16),
    ([5, 1100, 1, 1009, 1], 1, 128, 16),                  # units just above and below those a block takes whole
])
def test_a_long_sequence_among_short_ones(lens, Hkv, dh, page):
    kc, vc, bt = paged(lens, Hkv, dh, page, 73)
    q = synth.normal((len(lens), 4 * Hkv, dh), 73, 3, 1.0, "cuda")
    ro, rl = exact_on_gpu(q, kc, vc, bt, lens, page)
    got, lse = decode_one_layer(q, kc, vc, bt, lens, page)
    assert ((got - ro).norm(dim=(1, 2)) <= REL * ro.norm(dim=(1, 2))).all() and (lse - rl).abs().max() <= 2e-6


@pytest.mark.parametrize("first,second,Hkv,dh,page", [
    ([20000], [777], 1, 128, 128),                        # many shares, few
    ([300, 5000, 1100], [4000, 200, 129], 2, 128, 16),
    ([130] * 32, [130] * 31 + [9000], 2, 64, 16),         # whole units, shares
    ([700] * 33, [700] * 32 + [8000], 2, 64, 16),         # more lengths than a warp's lanes
])
def test_lengths_written_by_the_kernel_ahead(first, second, Hkv, dh, page):
    """The lengths are looked at before the kernel ahead has finished; what it writes counts.  It is the library's GEMM of one
    row, whose blocks let the next kernel come up as soon as they are set up, and which then takes tens of microseconds on
    eight SMs: its one-hot row picks a row of bf16 numbers whose bits are those of the lengths (from 128 on, all of them
    normal), in turn those of one list and the other's."""
    from paper_2608_15943_b200 import kvp
    longest = [max(a, b) for a, b in zip(first, second)]
    kc, vc, bt = paged(longest, Hkv, dh, page, 74)
    q = synth.normal((len(first), 4 * Hkv, dh), 74, 3, 1.0, "cuda")
    want = [exact_on_gpu(q, kc, vc, bt, lens, page) for lens in (first, second)]
    pad, K = -len(first) % 4, 1 << 17                      # 16-byte rows
    bits = torch.tensor([lens + [0] * pad for lens in (first, second)], dtype=torch.int32, device="cuda").view(torch.bfloat16)
    assert all(128 <= n < 32640 for n in first + second)
    table_of = torch.zeros(bits.shape[1], K, dtype=torch.bfloat16, device="cuda")
    table_of[:, 0], table_of[:, K - 1] = bits[0], bits[1]
    pick = torch.zeros(2, 1, K, dtype=torch.bfloat16, device="cuda")
    pick[0, 0, 0] = pick[1, 0, K - 1] = 1.0
    lengths = bits[1:].clone()
    desc = kvp.DecodeDesc(1, len(first), 4 * Hkv, Hkv, dh, page, bt.shape[1], kc.shape[0])
    ws = torch.empty(kvp.decode_workspace_bytes(desc, [0]), dtype=torch.uint8, device="cuda")
    table = bt.cuda()
    out = [(torch.full_like(q, float("nan")), torch.full(q.shape[:2], float("nan"), device="cuda")) for _ in range(20)]
    seen = [torch.empty_like(lengths) for _ in out]
    torch.cuda.synchronize()
    for i, (o, lse) in enumerate(out):
        kvp.gemm(pick[i % 2], table_of, lengths)
        kvp.decode(desc, [0], [q], [kc], [vc], table, lengths.view(torch.int32).view(-1)[:len(first)], [o], [lse], ws)
        seen[i].copy_(lengths)
    assert kvp.device_status() == kvp.OK
    for i, (o, lse) in enumerate(out):
        assert torch.equal(seen[i].view(torch.int32), bits[i % 2:i % 2 + 1].view(torch.int32))
        ro, rl = want[i % 2]
        assert (o.double() - ro).norm() <= REL * ro.norm() and (lse.double() - rl).abs().max() <= 2e-6, i
