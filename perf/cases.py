"""Performance cases of the library: what its users call, at the sizes they call it with.

A case is one call (or the pair of calls of a training step) through the public entry points of
`paper_2609_31093_b200`:

    forward          prefill: pyramid, routing and attention in one call, device tensors
    forward_host     the same for tensors that live in pinned host memory
    forward_packed   prefill of a variable-length batch
    select           block selection alone (pyramid + routing), what the paper's benchmark times
    decode           one generated token per sequence over a cached pyramid
    backward         attention backward for the indices a forward pass selected
    train_packed     forward and backward over a packed batch of documents

The head / block shapes are those of the repository's workloads (`SHAPES`); lengths run from a few hundred
tokens to 131072 and are not multiples of the block size as a rule.
"""
from __future__ import annotations

import math
import random

import torch

import paper_2609_31093_b200 as P
from paper_2609_31093_b200 import binding as PB

# (Hq, Hkv, d, C, g, K, dtype) of the repository's workloads
SHAPES = {
    "fp32_small": (1, 1, 64, 64, 2, 4, "fp32"),      # the tiny fp32 workload
    "mha16": (16, 16, 128, 64, 2, 16, "bf16"),       # one KV head per query head
    "gqa32_fan4": (32, 8, 128, 64, 4, 16, "bf16"),   # fan-in 4
    "gqa32_c128": (32, 8, 128, 128, 2, 32, "bf16"),  # the headline shape
    "gqa16": (16, 4, 128, 64, 2, 16, "bf16"),        # the scaling sweep
    "gqa32_d64": (32, 2, 64, 64, 2, 8, "bf16"),      # the paper's own benchmark shape
}

# what one call may cost at most: the listed cases' largest
_MAX_TOKENS = {"forward": 131072, "forward_host": 32768, "select": 131072, "backward": 32768,
               "forward_packed": 65536, "train_packed": 32768, "decode": 262144, "fp32": 4096}


def listed():
    return [
        # generation at long context, one user: the latency of one token
        dict(name="decode_128k", op="decode", shape="gqa32_c128", B=1, N=131072, pos=130037),
        # generation for a batch of users at ordinary context
        dict(name="decode_batch32_8k", op="decode", shape="gqa16", B=32, N=8192, pos=7777),
        # fp32 checks and small research models
        dict(name="forward_fp32_1k", op="forward", shape="fp32_small", B=1, N=1024),
        # a short prompt: launches and latency
        dict(name="forward_1500", op="forward", shape="gqa16", B=1, N=1500),
        # an ordinary prompt, one KV head per query head
        dict(name="forward_mha_8k", op="forward", shape="mha16", B=1, N=8192),
        # a batch of long prompts, fan-in 4, ragged end
        dict(name="forward_fan4_2x32k", op="forward", shape="gqa32_fan4", B=2, N=32700),
        # the headline workload
        dict(name="forward_128k", op="forward", shape="gqa32_c128", B=1, N=131072),
        # selection alone at the paper's benchmark shape
        dict(name="select_d64_64k", op="select", shape="gqa32_d64", B=1, N=65536),
        # prefill of many prompts of mixed length in one call
        dict(name="forward_packed_40", op="forward_packed", shape="gqa16", nseq=40, longest=4096, lengths=11),
        # a training step over packed documents
        dict(name="train_packed_12", op="train_packed", shape="gqa32_fan4", nseq=12, longest=6000, lengths=12),
        # attention backward of a long sequence
        dict(name="backward_32k", op="backward", shape="gqa32_c128", B=1, N=32768),
        # tensors in host memory: the copies are part of the call
        dict(name="forward_host_16k", op="forward_host", shape="gqa16", B=1, N=16384),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the call by how often it is made, the shape at random, the length over its logarithm."""
    op = rng.choices(["forward", "decode", "backward", "forward_packed", "select", "train_packed", "forward_host"],
                     weights=[6, 4, 3, 2, 2, 1, 1])[0]
    bf16 = [s for s in SHAPES if s != "fp32_small"]
    shape = rng.choice(bf16)
    top = _MAX_TOKENS[op]
    if op == "forward" and rng.random() < 0.15:
        shape, top = "fp32_small", _MAX_TOKENS["fp32"]
    if op in ("forward_packed", "train_packed"):
        nseq, longest = _log_int(rng, 3, 64), _log_int(rng, 200, 8192)
        return dict(op=op, shape=shape, nseq=min(nseq, max(3, top // longest)), longest=longest,
                    lengths=rng.randrange(1000))
    if op == "decode":
        N = _log_int(rng, 1024, top)
        B = min(_log_int(rng, 1, 64), max(1, 2 * top // N))
        return dict(op=op, shape=shape, B=B, N=N, pos=rng.randrange(N // 2, N))
    N = _log_int(rng, 256, top)
    if rng.random() < 0.25:
        N = max(256, N // 64 * 64)
    B = min(rng.choice([1, 1, 1, 2, 3, 4]), max(1, top // N))
    return dict(op=op, shape=shape, B=B, N=N)


# ------------------------------------------------------------------------------------------ inputs

def _lengths(case):
    """Sequence lengths of a packed batch: spread over their logarithm, one of them the longest."""
    rng = random.Random(case["lengths"])
    lens = [_log_int(rng, 16, case["longest"]) for _ in range(case["nseq"] - 1)] + [case["longest"]]
    rng.shuffle(lens)
    return lens


def _params(case, N=None, B=None):
    Hq, Hkv, d, C, g, K, dtype = SHAPES[case["shape"]]
    return P.Params(case.get("B", 1) if B is None else B, case["N"] if N is None else N, Hq, Hkv, d, C, g, K, dtype=dtype)


def _tensors(case, seed, B, N, starts=(0,)):
    """q, k, v as attention layers see them: unit noise; passages of a few hundred tokens whose keys and queries
    share one of 32 topic directions per KV head (a query finds its topic's blocks all over the context); and an
    attention sink, a first key of large norm along a direction that all queries share, with about half of a
    row's probability."""
    Hq, Hkv, d, C, g, K, dtype = SHAPES[case["shape"]]
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(int(seed) * 1000003 + 17)
    normal = lambda *s: torch.randn(s, generator=gen, device="cuda")  # noqa: E731
    G = Hq // Hkv
    passage = (torch.rand((B, N), generator=gen, device="cuda") < 1.0 / 400).cumsum(1)
    q = torch.empty((B, N, Hq, d), dtype=dt, device="cuda")
    k = torch.empty((B, N, Hkv, d), dtype=dt, device="cuda")
    v = torch.empty((B, N, Hkv, d), dtype=dt, device="cuda")
    sink_logit = math.log(K * C) + 0.5 + 0.25 * math.sqrt(d)
    for h in range(Hkv):
        topics = 0.5 * normal(32, d)
        which = torch.randint(0, 32, (N + 1,), generator=gen, device="cuda")[passage]
        mean = topics[which]                                               # [B, N, d]
        u = normal(d).sign()
        q[:, :, h * G:(h + 1) * G] = normal(B, N, G, d) + mean[:, :, None] + 0.3 * u
        k[:, :, h] = normal(B, N, d) + mean
        v[:, :, h] = normal(B, N, d)
        for s in starts:
            k[:, s, h] = sink_logit / (0.3 * math.sqrt(d)) * u + 0.3 * normal(B, d)
    return q, k, v


def prepare(case, seed):
    op = case["op"]
    Hq, Hkv, d, C, g, K, dtype = SHAPES[case["shape"]]
    s = {"op": op}
    if op in ("forward_packed", "train_packed"):
        lens = _lengths(case)
        cu = [0]
        for n in lens:
            cu.append(cu[-1] + n)
        total = cu[-1]
        p = _params(case, N=max(lens), B=1)
        q, k, v = (t[0] for t in _tensors(case, seed, 1, total, starts=cu[:-1]))
        s.update(p=p, cu=cu, q=q, k=k, v=v, pyramid=PB.alloc_pyramid(p), out=torch.zeros_like(q),
                 idx=torch.zeros(Hkv * K * total, dtype=torch.int32, device="cuda"),
                 lse=torch.zeros(Hq * total, dtype=torch.float32, device="cuda"),
                 ws=PB.alloc_workspace(p, PB.OP_FORWARD_PACKED))
        if op == "train_packed":
            s.update(dout=_dout(q, seed), dq=torch.zeros_like(q), dk=torch.zeros_like(k), dv=torch.zeros_like(v),
                     ws_bwd=PB.alloc_workspace(p, PB.OP_BSA_BWD_PACKED))
        return s
    B, N = case["B"], case["N"]
    p = _params(case)
    q, k, v = _tensors(case, seed, B, N)
    if op == "decode":
        pos = case["pos"]
        k[:, pos + 1:] = 0
        v[:, pos + 1:] = 0
        pyramid = PB.alloc_pyramid(p).zero_()
        P.pisa_build_pyramid(p, k, pyramid)
        s.update(p=p, pos=pos, q=q[:, pos].contiguous(), k=k, v=v, pyramid=pyramid,
                 idx=torch.zeros((B, Hkv, K), dtype=torch.int32, device="cuda"),
                 out=torch.zeros((B, Hq, d), dtype=q.dtype, device="cuda"),
                 lse=torch.zeros((B, Hq), dtype=torch.float32, device="cuda"), ws=PB.alloc_workspace(p, PB.OP_DECODE))
        return s
    if op == "forward_host":
        pin = lambda t: torch.empty(t.shape, dtype=t.dtype, pin_memory=True)  # noqa: E731
        s.update(p=p, q=pin(q).copy_(q), k=pin(k).copy_(k), v=pin(v).copy_(v), out=pin(q),
                 lse=torch.empty((B, Hq, N), dtype=torch.float32, pin_memory=True),
                 idx=torch.empty((B, Hkv, N, K), dtype=torch.int32, pin_memory=True),
                 ws=PB.alloc_workspace(p, PB.OP_FORWARD_HOST))
        return s
    pyramid = PB.alloc_pyramid(p).zero_()
    idx = torch.zeros((B, Hkv, N, K), dtype=torch.int32, device="cuda")
    if op == "select":
        s.update(p=p, q=q, k=k, pyramid=pyramid, idx=idx, ws=PB.alloc_workspace(p, PB.OP_ROUTE))
        return s
    out = torch.zeros_like(q)
    lse = torch.zeros((B, Hq, N), dtype=torch.float32, device="cuda")
    ws = PB.alloc_workspace(p, PB.OP_FORWARD)
    s.update(p=p, q=q, k=k, v=v, idx=idx, out=out, lse=lse)
    if op == "forward":
        s.update(pyramid=pyramid, ws=ws)
    else:
        P.pisa_forward(p, q, k, v, pyramid, idx, out, lse, ws)
        s.update(dout=_dout(q, seed), dq=torch.zeros_like(q), dk=torch.zeros_like(k), dv=torch.zeros_like(v),
                 ws=PB.alloc_workspace(p, PB.OP_BSA_BWD))
    return s


def _dout(q, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed) * 1000003 + 29)
    return torch.empty(q.shape, dtype=q.dtype, device="cuda").normal_(generator=gen)


# ------------------------------------------------------------------------------------------ one pass

def run(s):
    op = s["op"]
    if op == "forward":
        P.pisa_forward(s["p"], s["q"], s["k"], s["v"], s["pyramid"], s["idx"], s["out"], s["lse"], s["ws"])
        return {n: s[n] for n in ("out", "lse", "idx", "pyramid")}
    if op == "decode":
        P.pisa_decode_step(s["p"], s["pos"], s["q"], s["k"], s["v"], s["pyramid"], s["idx"], s["out"], s["lse"], s["ws"])
        return {n: s[n] for n in ("out", "lse", "idx", "pyramid")}
    if op == "select":
        P.pisa_build_pyramid(s["p"], s["k"], s["pyramid"])
        P.pisa_route(s["p"], s["q"], s["k"], s["pyramid"], s["idx"], None, s["ws"])
        return {n: s[n] for n in ("idx", "pyramid")}
    if op == "backward":
        P.pisa_bsa_bwd(s["p"], s["q"], s["k"], s["v"], s["idx"], s["out"], s["lse"], s["dout"], s["dq"], s["dk"],
                       s["dv"], s["ws"])
        return {n: s[n] for n in ("dq", "dk", "dv")}
    if op == "forward_host":
        P.pisa_forward_host(s["p"], s["q"], s["k"], s["v"], s["out"], s["lse"], s["idx"], s["ws"])
        return {n: s[n] for n in ("out", "lse", "idx")}
    P.pisa_forward_packed(s["p"], s["cu"], s["q"], s["k"], s["v"], s["pyramid"], s["idx"], s["out"], s["lse"], s["ws"])
    if op == "forward_packed":
        return {n: s[n] for n in ("out", "lse", "idx")}
    P.pisa_bsa_bwd_packed(s["p"], s["cu"], s["q"], s["k"], s["v"], s["idx"], s["out"], s["lse"], s["dout"], s["dq"],
                          s["dk"], s["dv"], s["ws_bwd"])
    return {n: s[n] for n in ("out", "lse", "idx", "dq", "dk", "dv")}


# ------------------------------------------------------------------------------------------ work

def _blocks(N, C, g, K, first=0):
    """Per leaf block c of a sequence: (its tokens, intermediate candidates scored, leaves scored, leaves kept)."""
    M = [N, -(-N // C)]
    while M[-1] > 1:
        M.append(-(-M[-1] // g))
    L = len(M) - 1
    for c in range(first, M[1]):
        inter = leaf = 0
        kept = 1
        for l in range(L, 0, -1):
            anc = c // g ** (l - 1)
            n = 1 if l == L else (kept - 1) * g + anc - c // g ** l * g + 1
            if n > K:
                scored = n - len({0, anc, max(c - 1, 0) // g ** (l - 1)})
                inter, leaf = (inter + scored, leaf) if l >= 2 else (inter, leaf + scored)
                kept = K
            else:
                kept = n
        yield min(C, N - c * C), inter, leaf, kept


def work(case):
    """Flops of the definition: a scored intermediate candidate costs g, a scored leaf C dot products per head, a
    kept leaf 2 C of them forward and 5 C backward.  Bytes: tensors in and out once (for decoding the rows that
    the selection and the attention of this one token read)."""
    Hq, Hkv, d, C, g, K, dtype = SHAPES[case["shape"]]
    op, es = case["op"], 2 if dtype == "bf16" else 4
    packed = op in ("forward_packed", "train_packed")
    lens, B = (_lengths(case), 1) if packed else ([case["N"]], case["B"])
    if op == "decode":
        _, inter, leaf, kept = next(_blocks(case["pos"] + 1, C, g, K, first=case["pos"] // C))
        rows = inter * g + leaf * C + 2 * kept * C
        return {"bytes": float(B * (Hkv * (rows * d * es + K * 4) + Hq * (2 * d * es + 4))),
                "flops": 2.0 * B * Hq * d * rows}
    tokens = B * sum(lens)
    select = attend = 0
    for n in lens:
        for t, inter, leaf, kept in _blocks(n, C, g, K):
            select += t * (inter * g + leaf * C)
            attend += t * kept * C
    per_dot = 2.0 * B * Hq * d
    qrow, krow, irow = Hq * d * es, Hkv * d * es, Hkv * K * 4
    forward_bytes = tokens * (2 * qrow + 2 * krow + irow + Hq * 4)
    backward_bytes = tokens * (4 * qrow + 4 * krow + irow + Hq * 4)
    if op == "select":
        return {"bytes": float(tokens * (qrow + krow + irow)), "flops": per_dot * select}
    if op == "backward":
        return {"bytes": float(backward_bytes), "flops": per_dot * 5 * attend}
    flops = per_dot * (select + 2 * attend)
    if op == "train_packed":
        return {"bytes": float(forward_bytes + backward_bytes), "flops": flops + per_dot * 5 * attend}
    return {"bytes": float(forward_bytes), "flops": flops}


def tolerance(case):
    """bf16: outputs, summaries and gradients are rounded to 8 bits (and so are the probabilities inside the
    products).  fp32: sums of up to K C terms; a row whose last kept and first dropped block tie to the last bits
    may take either, which changes that row's output a little.  The same goes for the share of indices."""
    if SHAPES[case["shape"]][6] == "fp32":
        return {"rel": 1e-4, "max": 0.1, "differ": 2e-3}
    return {"rel": 1e-2, "max": 0.4, "differ": 5e-3}
