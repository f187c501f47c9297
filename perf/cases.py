"""Performance cases: the work a user of the library has it do, through the Python binding of its C ABI.

Four kinds of call sequence, each over the range of sizes it is used at:

  block         projections and attention of a stack of layers, forward (prefill) or forward + backward (a training
                step), optionally with the output projection (the attention block of a pipeline stage)
  stage         forward pass of a decoder stage with real data flow from layer to layer (norms, rotary embedding,
                attention, gated MLP, residuals, optional LM head): a prompt or a training micro-batch
  stage_token   the same stage for one new token per sequence, layer by layer over the shared paged cache
  decode        cache append and split-KV decode attention of all layers of one step over the shared paged cache

Shapes come from the repository's workloads (paper_2608_15943_b200/workloads.py, bench.py) and tests, or are generic.
"""
import math
import random

import torch

from paper_2608_15943_b200 import kvp

BF, F32 = torch.bfloat16, torch.float32
DEV = "cuda"
THETA = 10000.0
EPS = 1e-5


# ---------------------------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------------------------
def block(name, L, B, S, D, Hq, Hkv, dh, share, backward, out_proj=False, fp32=False, causal=True):
    """share: the last `share` layers of the stack attend to the K/V of the layer before them."""
    return dict(name=name, kind="block", L=L, B=B, S=S, D=D, Hq=Hq, Hkv=Hkv, dh=dh, share=share, backward=backward,
                out_proj=out_proj, fp32=fp32, causal=causal)


def stage(name, L, B, S, D, Hq, Hkv, dh, F, V, share):
    return dict(name=name, kind="stage", L=L, B=B, S=S, D=D, Hq=Hq, Hkv=Hkv, dh=dh, F=F, V=V, share=share)


def stage_token(name, L, B, context, D, Hq, Hkv, dh, F, page, share):
    return dict(name=name, kind="stage_token", L=L, B=B, context=context, D=D, Hq=Hq, Hkv=Hkv, dh=dh, F=F, page=page, share=share)


def decode(name, L, B, lo, hi, Hq, Hkv, dh, page, pairs, fp32=False):
    """pairs: the last 2 * pairs layers share in pairs (an even layer's K/V serves the odd layer above it)."""
    return dict(name=name, kind="decode", L=L, B=B, lo=lo, hi=hi, Hq=Hq, Hkv=Hkv, dh=dh, page=page, pairs=pairs, fp32=fp32)


def listed():
    return [
        # the smallest training step: the tiny stack a user checks an integration with, fp32 tensors
        block("train-tiny-fp32", 4, 2, 128, 256, 4, 2, 64, 3, True, fp32=True),
        # fine-tuning a small model on sequences of no round length
        block("train-ragged", 3, 3, 776, 1024, 16, 4, 64, 1, True),
        # the long-sequence training step (eight layers, half of them on one donor)
        block("train-long", 8, 2, 8192, 4096, 32, 8, 128, 3, True),
        # prefill of a batch of 4K prompts
        block("prefill", 8, 4, 4096, 4096, 32, 8, 128, 3, False),
        # the attention block of a tail pipeline stage, one micro-batch, output projection included
        block("stage-block-train", 4, 8, 4096, 4096, 32, 8, 128, 3, True, out_proj=True),
        # one short prompt of odd length through a tail stage with its LM head
        stage("stage-prompt", 4, 1, 347, 4096, 32, 32, 128, 11008, 32000, 3),
        # a training micro-batch through the same stage
        stage("stage-microbatch", 4, 1, 8192, 4096, 32, 32, 128, 11008, 32000, 3),
        # serving: one token for each of 16 sequences through a stage
        stage_token("stage-token", 4, 16, 4096, 4096, 32, 8, 128, 11008, 128, 2),
        # the smallest decode step: the tiny stack, fp32 queries and outputs
        decode("decode-tiny-fp32", 4, 2, 129, 144, 4, 2, 64, 16, 2, fp32=True),
        # a small batch at moderate context
        decode("decode-small", 4, 8, 8192, 16384, 32, 8, 128, 128, 2),
        # the serving batch at long context (a quarter of the 32-layer stack), ragged lengths
        decode("decode-batch-long", 8, 32, 16384, 32768, 32, 8, 128, 128, 2),
        # few sequences at the longest context, one KV head per query head
        decode("decode-mha-128k", 2, 4, 122880, 131072, 32, 32, 128, 128, 1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


MAX_FLOPS = 4.0e13     # below the largest listed case
MAX_CACHE = 1.6e10     # bytes of K/V one decode case keeps


def draw(rng):
    kind = rng.choice(("block", "block", "stage", "stage_token", "decode", "decode"))
    dh = rng.choice((64, 128, 128))
    Hkv = rng.choice((2, 4, 8, 8))
    G = rng.choice((1, 2, 4, 4))
    if kind == "block":
        D = rng.choice((256, 512, 1024, 2048, 4096))
        L = rng.randint(1, 8)
        B = rng.randint(1, 4)
        S = _log_int(rng, 64, 8192)
        backward = rng.random() < 0.6
        fp32 = D <= 512 and B * S <= 2048 and rng.random() < 0.5
        c = block("", L, B, S, D, Hkv * G, Hkv, dh, rng.randint(0, L - 1), backward,
                  out_proj=not fp32 and rng.random() < 0.3, fp32=fp32, causal=rng.random() < 0.9)
    elif kind == "stage":
        D = rng.choice((1024, 2048, 4096))
        F = {1024: 2816, 2048: 5504, 4096: 11008}[D]
        L = rng.randint(1, 4)
        c = stage("", L, rng.randint(1, 4), _log_int(rng, 32, 4096), D, Hkv * G, Hkv, dh, F, rng.choice((0, 0, 32000)),
                  rng.randint(0, L - 1))
    elif kind == "stage_token":
        D = rng.choice((1024, 2048, 4096))
        F = {1024: 2816, 2048: 5504, 4096: 11008}[D]
        L = rng.randint(1, 4)
        c = stage_token("", L, _log_int(rng, 1, 64), _log_int(rng, 128, 16384), D, Hkv * G, Hkv, dh, F,
                        rng.choice((16, 64, 128)), rng.randint(0, L - 1))
    else:
        L = rng.randint(1, 8)
        lo = _log_int(rng, 128, 65536)
        c = decode("", L, _log_int(rng, 1, 32), lo, int(lo * rng.uniform(1.0, 2.0)), Hkv * G, Hkv, dh,
                   rng.choice((16, 32, 64, 128)), rng.randint(0, L // 2))
    while work(c)["flops"] > MAX_FLOPS or cache_bytes(c) > MAX_CACHE:
        if c["kind"] == "decode":
            c["lo"], c["hi"] = c["lo"] * 2 // 3, c["hi"] * 2 // 3
        elif c["kind"] == "stage_token":
            c["context"] = c["context"] * 2 // 3
        else:
            c["S"] = c["S"] * 2 // 3
    if c["kind"] == "block" and c["backward"]:
        step = 8 // math.gcd(8, c["B"])          # the weight gradients take B * S in multiples of 8
        c["S"] = max(step, c["S"] // step * step)
    del c["name"]
    return c


def donors(c):
    L = c["L"]
    if c["kind"] == "decode":
        first = L - 2 * c["pairs"]
        return [l if l < first or (l - first) % 2 == 0 else l - 1 for l in range(L)]
    d = L - 1 - c["share"]
    return [min(l, d) for l in range(L)]


def owners(c):
    return [l for l, d in enumerate(donors(c)) if d == l]


def cache_bytes(c):
    if c["kind"] == "decode":
        tokens = c["B"] * (c["lo"] + c["hi"]) / 2
    elif c["kind"] == "stage_token":
        tokens = c["B"] * c["context"]
    else:
        return 0
    return tokens * len(owners(c)) * 2 * c["Hkv"] * c["dh"] * 2


# ---------------------------------------------------------------------------------------------
# inputs and buffers
# ---------------------------------------------------------------------------------------------
class _Rand:
    def __init__(self, seed):
        self.g = torch.Generator(device=DEV).manual_seed(seed)
        self.host = random.Random(seed)

    def normal(self, *shape, std=1.0, fp32=False):
        t = torch.empty(*shape, device=DEV, dtype=BF).normal_(0.0, std, generator=self.g)
        return t.float() if fp32 else t


def _empty(*shape, dtype=BF):
    return torch.empty(*shape, device=DEV, dtype=dtype)


def _rows(stacked, layers, L):
    """Per-layer list over a stacked tensor: one row for each layer in `layers`, None elsewhere."""
    out = [None] * L
    for i, l in enumerate(layers):
        out[l] = stacked[i]
    return out


def _prepare_block(c, seed):
    r = _Rand(seed)
    L, B, S, D, Hq, Hkv, dh, fp32 = (c[k] for k in ("L", "B", "S", "D", "Hq", "Hkv", "dh", "fp32"))
    T, nq, nkv, own, every = B * S, Hq * dh, Hkv * dh, owners(c), range(L)
    dt = F32 if fp32 else BF
    donor = donors(c)
    sh = kvp.Shape(L, B, S, D, Hq, Hkv, dh, kvp.F32 if fp32 else kvp.BF16)
    s = dict(kind="block", case=c, sh=sh, donor=donor)
    ins = dict(x=(every, (T, D), 1.0), wq=(every, (nq, D), 0.02), wk=(own, (nkv, D), 0.02), wv=(own, (nkv, D), 0.02))
    outs = dict(q=(every, (B, S, Hq, dh), dt), k=(own, (B, S, Hkv, dh), dt), v=(own, (B, S, Hkv, dh), dt),
                o=(every, (B, S, Hq, dh), dt), lse=(every, (B, Hq, S), F32))
    if c["out_proj"]:
        ins["wo"] = (every, (D, nq), 0.02)
        outs["y"] = (every, (T, D), BF)
    if c["backward"]:
        if c["out_proj"]:
            ins["dy"] = (every, (T, D), 1.0)
            outs["d_o"] = (every, (B, S, Hq, dh), BF)
            outs["dwo"] = (every, (D, nq), F32)
        else:
            ins["d_o"] = (every, (B, S, Hq, dh), 1.0)
        outs.update(dq=(every, (B, S, Hq, dh), dt), dk_sum=(own, (B, S, Hkv, dh), F32), dv_sum=(own, (B, S, Hkv, dh), F32),
                    dwq=(every, (nq, D), F32), dwk=(own, (nkv, D), F32), dwv=(own, (nkv, D), F32), dx=(every, (T, D), dt))
    for name, (layers, shape, std) in ins.items():
        s[name] = _rows(r.normal(len(layers), *shape, std=std, fp32=fp32), layers, L)
    whole = {}
    for name, (layers, shape, dtype) in outs.items():
        whole[name] = _empty(len(layers), *shape, dtype=dtype)
        s[name] = _rows(whole[name], layers, L)
    s["outputs"] = whole
    ops = [kvp.OP_PROJ_FWD, kvp.OP_ATTN_FWD] + ([kvp.OP_ATTN_BWD, kvp.OP_PROJ_BWD] if c["backward"] else [])
    s["ws"] = _empty(max([256] + [kvp.workspace_bytes(op, sh, donor) for op in ops]), dtype=torch.uint8)
    return s


def _run_block(s):
    c, sh, donor, ws = s["case"], s["sh"], s["donor"], s["ws"]
    kvp.proj_fwd(sh, donor, s["x"], s["wq"], s["wk"], s["wv"], s["q"], s["k"], s["v"], ws)
    kvp.attn_fwd(sh, donor, s["q"], s["k"], s["v"], s["o"], s["lse"], causal=c["causal"], ws=ws)
    if c["out_proj"]:
        kvp.out_proj_fwd(sh, s["o"], s["wo"], s["y"])
    if c["backward"]:
        if c["out_proj"]:
            kvp.out_proj_bwd(sh, s["o"], s["wo"], s["dy"], s["d_o"], s["dwo"])
        kvp.attn_bwd(sh, donor, s["q"], s["k"], s["v"], s["o"], s["d_o"], s["lse"], s["dq"], s["dk_sum"], s["dv_sum"], ws,
                     causal=c["causal"])
        kvp.proj_bwd(sh, donor, s["x"], s["wq"], s["wk"], s["wv"], s["dq"], s["dk_sum"], s["dv_sum"], s["dwq"], s["dwk"],
                     s["dwv"], s["dx"], ws)
    return s["outputs"]


def _layer_weights(c, r):
    """Weights of each layer of a decoder stage; K/V projections on owners only."""
    D, F, nq, nkv, own = c["D"], c["F"], c["Hq"] * c["dh"], c["Hkv"] * c["dh"], owners(c)
    w = []
    for l in range(c["L"]):
        m = dict(n1=1.0 + r.normal(D, std=0.1), n2=1.0 + r.normal(D, std=0.1), wq=r.normal(nq, D, std=0.02),
                 wo=r.normal(D, nq, std=0.02), gate=r.normal(F, D, std=0.02), up=r.normal(F, D, std=0.02),
                 down=r.normal(D, F, std=0.02))
        if l in own:
            m.update(wk=r.normal(nkv, D, std=0.02), wv=r.normal(nkv, D, std=0.02))
        w.append(m)
    return w


def _stage_buffers(s, c, T):
    D, F, nq = c["D"], c["F"], c["Hq"] * c["dh"]
    s.update(n=_empty(T, D), q=_empty(T, nq), o=_empty(T, nq), y=_empty(T, D), mid=_empty(T, D), gate=_empty(T, F),
             up=_empty(T, F), out=[_empty(T, D) for _ in range(c["L"])])


def _prepare_stage(c, seed):
    r = _Rand(seed)
    B, S, D, Hkv, dh, V = (c[k] for k in ("B", "S", "D", "Hkv", "dh", "V"))
    T = B * S
    s = dict(kind="stage", case=c, donor=donors(c), sh=kvp.Shape(1, B, S, D, c["Hq"], Hkv, dh), h=r.normal(T, D),
             w=_layer_weights(c, r))
    _stage_buffers(s, c, T)
    s["lse"] = _empty(B, c["Hq"], S, dtype=F32)
    s["k"] = {l: _empty(B, S, Hkv, dh) for l in owners(c)}
    s["v"] = {l: _empty(B, S, Hkv, dh) for l in owners(c)}
    if V:
        s.update(n_last=1.0 + r.normal(D, std=0.1), lm=r.normal(V, D, std=0.02), logits=_empty(T, V))
    return s


def _project(s, sh, l, k, v):
    """Q of layer l into s["q"]; an owner projects its K and V too (one call), a consumer only its queries."""
    m = s["w"][l]
    if s["donor"][l] == l:
        kvp.proj_fwd(sh, [0], [s["n"]], [m["wq"]], [m["wk"]], [m["wv"]], [s["q"]], [k], [v])
    else:
        kvp.gemm(s["n"], m["wq"], s["q"])


def _after_attention(s, l, x):
    """Output projection, residual, norm, gated MLP, residual of layer l; returns the residual stream."""
    m = s["w"][l]
    kvp.gemm(s["o"], m["wo"], s["y"])
    kvp.add(x, s["y"], s["mid"])
    kvp.rmsnorm(s["mid"], m["n2"], EPS, s["n"])
    kvp.gemm(s["n"], m["gate"], s["gate"])
    kvp.gemm(s["n"], m["up"], s["up"])
    kvp.swiglu(s["gate"], s["up"], s["gate"])
    kvp.gemm(s["gate"], m["down"], s["y"])
    return kvp.add(s["mid"], s["y"], s["out"][l])


def _run_stage(s):
    c, sh, x = s["case"], s["sh"], s["h"]
    B, S, Hq, dh = c["B"], c["S"], c["Hq"], c["dh"]
    q, o = s["q"].view(B, S, Hq, dh), s["o"].view(B, S, Hq, dh)
    for l, d in enumerate(s["donor"]):
        kvp.rmsnorm(x, s["w"][l]["n1"], EPS, s["n"])
        _project(s, sh, l, s["k"].get(l), s["v"].get(l))
        kvp.rope(q, THETA)
        if d == l:
            kvp.rope(s["k"][l], THETA)
        kvp.attn_fwd(sh, [0], [q], [s["k"][d]], [s["v"][d]], [o], [s["lse"]])
        x = _after_attention(s, l, x)
    out = dict(x=x, k=s["k"], v=s["v"])
    if c["V"]:
        kvp.rmsnorm(x, s["n_last"], EPS, s["n"])
        out["logits"] = kvp.gemm(s["n"], s["lm"], s["logits"])
    return out


def _paged_cache(c, r, lengths, longest, page):
    """Pools of the owner layers, filled; the pages of the sequences lie scattered over the pool."""
    need = [(n + page - 1) // page for n in lengths]
    n_pages = len(lengths) * ((longest + page - 1) // page)
    max_pages = (longest + 256 + page - 1) // page           # room for the sequences to grow
    order = list(range(n_pages))
    r.host.shuffle(order)
    table = torch.zeros(len(lengths), max_pages, dtype=torch.int32)
    at = 0
    for b, n in enumerate(need):
        table[b, :n] = torch.tensor(order[at:at + n], dtype=torch.int32)
        at += n
    own = owners(c)
    kc = _rows([r.normal(n_pages, c["Hkv"], page, c["dh"]) for _ in own], own, c["L"])
    vc = _rows([r.normal(n_pages, c["Hkv"], page, c["dh"]) for _ in own], own, c["L"])
    return dict(kc=kc, vc=vc, table=table.to(DEV), lengths=torch.tensor(lengths, dtype=torch.int32, device=DEV),
                max_pages=max_pages, n_pages=n_pages)


def _prepare_stage_token(c, seed):
    r = _Rand(seed)
    B, D, Hq, Hkv, dh, page = (c[k] for k in ("B", "D", "Hq", "Hkv", "dh", "page"))
    s = dict(kind="stage_token", case=c, donor=donors(c), sh=kvp.Shape(1, B, 1, D, Hq, Hkv, dh), h=r.normal(B, D),
             w=_layer_weights(c, r))
    _stage_buffers(s, c, B)
    s.update(_paged_cache(c, r, [c["context"]] * B, c["context"], page))     # sequences that advance together
    s["desc"] = kvp.DecodeDesc(1, B, Hq, Hkv, dh, page, s["max_pages"], s["n_pages"])
    s["ws"] = _empty(max(256, kvp.decode_workspace_bytes(s["desc"], [0])), dtype=torch.uint8)
    s.update(lse=_empty(B, Hq, dtype=F32), k_new=_empty(B, Hkv, dh), v_new=_empty(B, Hkv, dh))
    return s


def _run_stage_token(s):
    c, sh, desc, x = s["case"], s["sh"], s["desc"], s["h"]
    B, Hq, Hkv, dh, pos = c["B"], c["Hq"], c["Hkv"], c["dh"], c["context"] - 1
    q, o = s["q"].view(B, Hq, dh), s["o"].view(B, Hq, dh)
    for l, d in enumerate(s["donor"]):
        kvp.rmsnorm(x, s["w"][l]["n1"], EPS, s["n"])
        _project(s, sh, l, s["k_new"], s["v_new"])
        kvp.rope(q.view(B, 1, Hq, dh), THETA, pos)
        if d == l:
            kvp.rope(s["k_new"].view(B, 1, Hkv, dh), THETA, pos)
            kvp.cache_append(desc, [0], [s["k_new"]], [s["v_new"]], [s["kc"][l]], [s["vc"][l]], s["table"], s["lengths"])
        kvp.decode(desc, [0], [q], [s["kc"][d]], [s["vc"][d]], s["table"], s["lengths"], [o], [s["lse"]], s["ws"])
        x = _after_attention(s, l, x)
    return dict(x=x, kc=s["kc"], vc=s["vc"])


def _prepare_decode(c, seed):
    r = _Rand(seed)
    L, B, Hq, Hkv, dh, page, fp32 = (c[k] for k in ("L", "B", "Hq", "Hkv", "dh", "page", "fp32"))
    donor, own = donors(c), owners(c)
    s = dict(kind="decode", case=c, donor=donor)
    s.update(_paged_cache(c, r, [r.host.randint(c["lo"], c["hi"]) for _ in range(B)], c["hi"], page))
    s["desc"] = kvp.DecodeDesc(L, B, Hq, Hkv, dh, page, s["max_pages"], s["n_pages"], 0, kvp.F32 if fp32 else kvp.BF16)
    s["ws"] = _empty(max(256, kvp.decode_workspace_bytes(s["desc"], donor)), dtype=torch.uint8)
    s["q"] = list(r.normal(L, B, Hq, dh, fp32=fp32))
    s["k_new"] = _rows(r.normal(len(own), B, Hkv, dh, fp32=fp32), own, L)
    s["v_new"] = _rows(r.normal(len(own), B, Hkv, dh, fp32=fp32), own, L)
    s["o_all"], s["lse_all"] = _empty(L, B, Hq, dh, dtype=F32 if fp32 else BF), _empty(L, B, Hq, dtype=F32)
    s["o"], s["lse"] = list(s["o_all"]), list(s["lse_all"])
    return s


def _run_decode(s):
    kvp.cache_append(s["desc"], s["donor"], s["k_new"], s["v_new"], s["kc"], s["vc"], s["table"], s["lengths"])
    kvp.decode(s["desc"], s["donor"], s["q"], s["kc"], s["vc"], s["table"], s["lengths"], s["o"], s["lse"], s["ws"])
    return dict(o=s["o_all"], lse=s["lse_all"], kc=s["kc"], vc=s["vc"])


def prepare(case, seed):
    return {"block": _prepare_block, "stage": _prepare_stage, "stage_token": _prepare_stage_token,
            "decode": _prepare_decode}[case["kind"]](case, seed)


def run(state):
    return {"block": _run_block, "stage": _run_stage, "stage_token": _run_stage_token,
            "decode": _run_decode}[state["kind"]](state)


# ---------------------------------------------------------------------------------------------
# work and tolerance
# ---------------------------------------------------------------------------------------------
def work(case):
    """Each input read once, each output written once (a decode step reads the stored K/V rows of its sequences once
    per donor and writes the new token's); a MAC counts 2, causal attention the visible pairs, backward twice forward."""
    c = case
    L, B, Hq, Hkv, dh, n_own = c["L"], c["B"], c["Hq"], c["Hkv"], c["dh"], len(owners(c))
    nq, nkv = Hq * dh, Hkv * dh
    if c["kind"] == "decode":
        e = 4 if c["fp32"] else 2
        flops = L * B * (c["lo"] + c["hi"]) / 2 * 4 * nq
        new = n_own * B * 2 * nkv
        return {"bytes": cache_bytes(c) + L * B * (2 * nq * e + Hq * 4) + new * (e + 2), "flops": flops}
    D = c["D"]
    if c["kind"] == "block":
        T, S, e = B * c["S"], c["S"], 4 if c["fp32"] else 2
        pairs = S * (S + 1) / 2 if c["causal"] else S * S
        proj = L * 2 * T * D * nq + n_own * 4 * T * D * nkv + (L * 2 * T * D * nq if c["out_proj"] else 0)
        fwd = proj + L * 4 * dh * pairs * B * Hq
        w = L * nq * D + n_own * 2 * nkv * D
        act = L * T * (D + 2 * nq) + n_own * T * 2 * nkv
        nbytes = (w + act) * e + L * T * Hq * 4
        if c["out_proj"]:
            nbytes += (L * D * nq + L * T * D) * e
        if c["backward"]:
            nbytes += (L * T * (nq + D) + L * T * (D + nq if c["out_proj"] else nq)) * e   # dq, dx; dy and d_o, or d_o
            nbytes += n_own * T * 2 * nkv * 4 + w * 4 + (L * D * nq * 4 if c["out_proj"] else 0)
        return {"bytes": nbytes, "flops": fwd * (3 if c["backward"] else 1)}
    T = B * (c["S"] if c["kind"] == "stage" else 1)
    w = L * (2 * nq * D + 3 * c["F"] * D) + n_own * 2 * nkv * D
    flops, nbytes = 2 * T * w, 2 * (w + 2 * L * D + 2 * T * D)
    if c["kind"] == "stage":
        flops += L * 4 * dh * c["S"] * (c["S"] + 1) / 2 * B * Hq + 2 * T * D * c["V"]
        nbytes += 2 * (c["V"] * D + T * c["V"] + n_own * T * 2 * nkv)
    else:
        flops += L * B * c["context"] * 4 * nq
        nbytes += cache_bytes(c)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """bf16 storage and bf16 tensor-core operands with fp32 accumulation, the fp32 interface included.  About four times
    what the path differs by from the same chain in 64 bits without intermediate roundings (2-norm): decode outputs
    2.2e-3, a block's outputs and gradients up to 3.4e-3; four layers of a stage 1.2e-2 (2.5 times that is stated)."""
    return {"rel": {"decode": 8e-3, "block": 1.3e-2, "stage": 3e-2, "stage_token": 3e-2}[case["kind"]]}
