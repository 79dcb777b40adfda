"""Keys, queries, values and gradients that are not finite: what they reach and what they must not.

Selection: a score that is not a number ranks after every other one, ties to the smaller index, on every path; a row always
gets min(K, leaves before it) distinct blocks, the forced ones among them."""
import math

import numpy as np
import pytest
import torch

import pisa_synth as S
from oracle import pisa_oracle as O

pytestmark = pytest.mark.gpu

import pisa_testlib as T  # noqa: E402
import paper_2609_31093_b200 as P  # noqa: E402
from paper_2609_31093_b200 import binding as PB  # noqa: E402

NAN = float("nan")


def _walk(q, k, level, M, L, C, g, K, pos):
    """Select_K of Sec. 3.2 for one row: q [G, d], k [N, d], level(l) [M_l, d] (device tensors).  Returns the leaves and the
    smallest relative gap between a kept and a dropped score (rows inside the tie band may go either way)."""
    q = q.double()
    scale = 1.0 / math.sqrt(q.shape[1])
    c = pos // C
    A, gap = [0], math.inf
    for l in range(L, 0, -1):
        V = [i for i in A if i < M[l] and i <= c // g ** (l - 1)]
        if len(V) > K:
            F = O.forced_nodes(l, c, g)
            rest = [i for i in V if i not in F]
            u = {}
            for i in rest:
                x = (k[i * C:(i + 1) * C] if l == 1 else level(l - 1)[i * g:(i + 1) * g]).double()
                s = float(torch.logsumexp(q @ x.T * scale, 1).sum())
                u[i] = -math.inf if math.isnan(s) else s
            order = sorted(rest, key=lambda i: (-u[i], i))
            keep = K - len(F)
            a, b = u[order[keep - 1]], u[order[keep]]
            if a > -math.inf:
                gap = min(gap, (a - b) / max(abs(a), 1.0))
            V = sorted(set(F) | set(order[:keep]))
        A = V if l == 1 else [r for i in V for r in range(i * g, i * g + g)]
    return A, gap


def _check_row(row, want, gap, K, c, what):
    n = min(K, c + 1)
    row = row.tolist()
    assert row[n:] == [-1] * (K - n) and all(a < b for a, b in zip(row[:n], row[1:n])), (what, row)
    assert {0, max(c - 1, 0), c} <= set(row[:n]) and 0 <= row[0] and row[n - 1] <= c, (what, row)
    if gap > T.TIE_BAND:
        assert row[:n] == want, (what, row, want)


@pytest.mark.parametrize("C,g,K,G", [(64, 2, 16, 4), (32, 4, 32, 1), (64, 4, 32, 16), (64, 4, 3, 2)])
def test_decoding_with_keys_that_are_not_numbers(C, g, K, G):
    N, Hkv, d = 8192, 2, 64
    w = S.Workload("nf_dec", 1, N, G * Hkv, Hkv, d, C, g, K, "bf16", 2100 + K, "iid")
    t = S.make_inputs(w)
    q, k, v = (T.to_torch(t[x], "bf16") for x in ("q", "k", "v"))
    rng = np.random.default_rng(5)
    M1 = N // C
    for leaf in rng.choice(np.arange(1, M1 - 3), size=M1 // 2, replace=False):       # half of all leaves
        k[0, int(leaf) * C + int(rng.integers(C)), 0] = NAN
    k[0, (M1 // 2) * C + 5, 1] = NAN                                                 # head 1: one leaf
    p = P.Params(1, N, G * Hkv, Hkv, d, C, g, K, dtype="bf16")
    pyr = PB.alloc_pyramid(p)
    P.pisa_build_pyramid(p, k, pyr)
    L, M, off, _ = P.pyramid_layout(p)
    ws = PB.alloc_workspace(p, PB.OP_DECODE)
    idx = torch.full((1, Hkv, K), -7, dtype=torch.int32, device="cuda")
    out, lse = torch.zeros((1, G * Hkv, d), dtype=torch.bfloat16, device="cuda"), torch.zeros((1, G * Hkv), device="cuda")
    for pos in (N - 1, N - 100, N // 2 + 3):
        P.pisa_decode_step(p, pos, q[:, pos].contiguous(), k, v, pyr, idx, out, lse, ws)
        torch.cuda.synchronize()
        assert P.read_status(ws) == 0
        for h in range(Hkv):
            level = lambda l: pyr[off[l]:off[l] + Hkv * M[l] * d].view(Hkv, M[l], d)[h]  # noqa: E731
            want, gap = _walk(q[0, pos, h * G:(h + 1) * G], k[0, :, h], level, M, L, C, g, K, pos)
            _check_row(idx[0, h], want, gap, K, pos // C, (pos, h))


@pytest.mark.parametrize("dtype,impl,N,C,g,K,G", [("bf16", PB.IMPL_SIMT, 6000, 64, 2, 16, 2), ("fp32", PB.IMPL_AUTO, 3000, 32, 4, 32, 1),
                                                  ("bf16", PB.IMPL_AUTO, 9000, 64, 2, 4, 16)])
def test_ranked_selections_with_keys_that_are_not_numbers(dtype, impl, N, C, g, K, G):
    """The kernels that select with a warp per token (SIMT; lists with large groups)."""
    _selection(dtype, impl, N, C, g, K, G)


@pytest.mark.parametrize("N,C,g,K,G", [(5000, 64, 2, 16, 4), (2500, 128, 4, 4, 2), (3000, 64, 4, 32, 1),   # query-major
                                       (20000, 64, 2, 16, 4), (9000, 64, 4, 8, 2)])                    # lists
def test_sorted_selections_with_keys_that_are_not_numbers(N, C, g, K, G):
    """The kernels that select with a thread per token and a sorting network."""
    _selection("bf16", PB.IMPL_AUTO, N, C, g, K, G)


def _selection(dtype, impl, N, C, g, K, G):
    Hkv, d = 2, 64
    w = S.Workload("nf_sel", 1, N, G * Hkv, Hkv, d, C, g, K, dtype, 2200 + K, "iid")
    t = S.make_inputs(w)
    dev = T.Device(w, t, impl=impl)
    rng = np.random.default_rng(6)
    M1 = -(-N // C)
    for leaf in rng.choice(np.arange(1, M1 - 3), size=M1 // 2, replace=False):
        dev.k[0, int(leaf) * C + int(rng.integers(C)), 0] = NAN
    dev.k[0, (M1 // 2) * C + 5, 1] = NAN
    dev.build_pyramid()
    dev.route(with_margin=False)
    assert dev.sync_status() == 0
    rows = sorted({0, C, K * C, N // 2 + 3, N - 1} | {int(x) for x in rng.integers(0, N, 20)})
    for h in range(Hkv):
        for pos in rows:
            want, gap = _walk(dev.q[0, pos, h * G:(h + 1) * G], dev.k[0, :, h], lambda l: dev.level(l)[0, h], dev.M, dev.L, C, g, K, pos)
            _check_row(dev.idx[0, h, pos], want, gap, K, pos // C, (pos, h))


def _see(idx, N, C, key):
    """Rows [B, Hkv, N] that selected the key's leaf and come no earlier than the key."""
    t = torch.arange(N, device="cuda")
    return (idx == key // C).any(-1) & (t >= key)


@pytest.mark.parametrize("N,G", [(300, 1), (700, 2), (1500, 1), (3000, 1), (700, 4)])      # eight, four and one warp per token
@pytest.mark.parametrize("what", ["k", "v"])
def test_fp32_rows_show_what_they_attend_to(N, G, what):
    """A NaN key or value reaches every row that selected and may see it, and no other one."""
    C, K = 64, 4
    w = S.Workload("nf_simt", 1, N, G, 1, 64, C, 2, K, "fp32", 2300 + N, "iid")
    dev = T.Device(w, S.make_inputs(w))
    dev.forward()
    assert dev.sync_status() == 0
    clean, idx = dev.out.clone(), dev.idx.clone()
    for keys in ([70], list(range(64, 128)), list(range(N - 20, N))):          # one key; a whole leaf; the last ones
        getattr(dev, what)[0, keys] = NAN
        dev.bsa(idx)
        assert dev.sync_status() == 0
        see = torch.stack([_see(idx, N, C, k)[0, 0] for k in keys]).any(0)
        assert bool(torch.isnan(dev.out[0, see]).all()), keys
        assert torch.equal(dev.out[0, ~see], clean[0, ~see]), keys
        dev = T.Device(w, S.make_inputs(w))


@pytest.mark.parametrize("B,G,C", [(1, 4, 64), (1, 16, 128), (40, 1, 32), (3, 8, 64)])
def test_decoding_shows_what_it_attends_to(B, G, C):
    """A NaN key or value of a selected block reaches the output, also where all keys of a warp's share are NaN; keys with
    logits of -inf weigh nothing."""
    N, K, Hkv, d, pos = 16 * C, 16, 2, 64, 16 * C - 5
    gen = torch.Generator(device="cuda").manual_seed(9)
    q, k, v = (torch.randn(s, generator=gen, device="cuda").bfloat16() for s in ((B, G * Hkv, d), (B, N, Hkv, d), (B, N, Hkv, d)))
    p = P.Params(B, N, G * Hkv, Hkv, d, C, 2, K, dtype="bf16")
    pyr, ws = PB.alloc_pyramid(p), PB.alloc_workspace(p, PB.OP_DECODE)
    P.pisa_build_pyramid(p, k, pyr)

    def step(kk, vv):
        idx = torch.full((B, Hkv, K), -7, dtype=torch.int32, device="cuda")
        out, lse = torch.zeros_like(q), torch.zeros((B, G * Hkv), device="cuda")
        P.pisa_decode_step(p, pos, q, kk, vv, pyr.clone(), idx, out, lse, ws)
        torch.cuda.synchronize()
        assert P.read_status(ws) == 0 and bool((idx == torch.arange(K, device="cuda", dtype=torch.int32)).all())
        return out, lse

    clean = step(k, v)
    for keys in (slice(7, 8), slice(3 * C, 4 * C), slice(0, N), slice(pos, pos + 1)):
        kk, vv = k.clone(), v.clone()
        kk[:, keys, 0] = NAN
        vv[:, keys, 1, 3] = NAN
        out, lse = step(kk, v)
        assert bool(torch.isnan(out[:, :G]).all()) and bool(torch.isnan(lse[:, :G]).all()), keys
        assert torch.equal(out[:, G:], clean[0][:, G:]) and torch.equal(lse[:, G:], clean[1][:, G:])
        out, lse = step(k, vv)
        assert bool(torch.isnan(out[:, G:, 3]).all()) and torch.equal(lse, clean[1])
        out[:, G:, 3] = clean[0][:, G:, 3]
        assert torch.equal(out, clean[0])
    if G == 1:
        kk = k.clone()
        gone = torch.zeros(N, dtype=torch.bool, device="cuda")
        gone[3 * C:5 * C] = True
        gone[:9] = True
        for h in range(Hkv):
            kk[:, gone, h] = torch.where(q[:, None, h] > 0, -math.inf, math.inf).bfloat16().expand(-1, int(gone.sum()), -1)
        out, lse = step(kk, v)
        z = torch.einsum("bhd,bnhd->bhn", q.float(), k.float()) * d ** -0.5
        z[:, :, gone] = -math.inf
        z[:, :, pos + 1:] = -math.inf
        want = torch.einsum("bhn,bnhd->bhd", torch.softmax(z, 2), v.float())
        assert float((out.float() - want).abs().max()) <= T.BF16_MAX_ABS and torch.allclose(lse, torch.logsumexp(z, 2), atol=1e-3)


def _poison(x, what, N, C):
    """x [B, N, H, d]"""
    H = x.shape[2]
    if what == "future":                          # everything from the middle of a leaf on
        x[:, N // 2 + 9:] = NAN
    elif what == "future_inf":                    # ... from a leaf's start on
        x[:, N // 2 // C * C:] = math.inf
    elif what == "key":                           # one key in the past of most rows, one column
        x[:, N // 3, 0, 5] = NAN
        x[:, N // 3 + C, H - 1, 7] = -math.inf
    else:                                         # a whole leaf, and the first leaf of the last batch element
        x[:, N // 3 // C * C:N // 3 // C * C + C] = NAN
        x[-1, :C, 0] = math.inf


def _same(got, want, what):
    """NaN (or infinite) where the reference is, equal to bf16 rounding elsewhere."""
    bad = ~torch.isfinite(want)
    assert torch.equal(~torch.isfinite(got), bad), (what, int((~torch.isfinite(got) & ~bad).sum()), int((torch.isfinite(got) & bad).sum()))
    g, w = got[~bad].double(), want[~bad].double()
    assert bool(((g - w).abs() <= 2.0 ** -6 * w.abs() + T.BF16_MAX_ABS).all()), what


FORWARD = [(2, 1500, 8, 2, 128, 64, 2, 4), (1, 700, 2, 2, 64, 64, 4, 4), (1, 900, 16, 1, 128, 128, 2, 3), (4, 2200, 32, 8, 64, 64, 2, 5),
           (1, 600, 4, 1, 64, 128, 4, 3)]


@pytest.mark.parametrize("shape", FORWARD, ids=lambda s: "b%d_n%d_h%d_%d_d%d_c%d_g%d_k%d" % s)
@pytest.mark.parametrize("tensor", ["k", "v", "q"])
@pytest.mark.parametrize("what", ["future", "future_inf", "key", "leaf"])
def test_dense_forward_shows_what_its_rows_selected(shape, tensor, what):
    """The dense tiles against the exact path (a warp per token, selected and visible keys only) on the same blocks."""
    B, N, Hq, Hkv, d, C, g, K = shape
    w = S.Workload("nf_fwd", B, N, Hq, Hkv, d, C, g, K, "bf16", 2400 + N, "iid")
    dev = T.Device(w, S.make_inputs(w))
    _poison(getattr(dev, tensor), what, N, C)
    dev.forward()
    assert dev.sync_status() == 0
    ref = T.Device(w, S.make_inputs(w), impl=PB.IMPL_SIMT)
    ref.q, ref.k, ref.v = dev.q, dev.k, dev.v
    ref.bsa(dev.idx)
    assert ref.sync_status() == 0
    _same(dev.out, ref.out, (tensor, what))
    ok = torch.isfinite(ref.lse)                  # (a NaN denominator reads -inf there)
    assert torch.allclose(dev.lse[ok], ref.lse[ok], rtol=1e-4, atol=1e-3)
    # a row whose past (up to its own token) is finite is what it was, and so are its blocks
    dev2 = T.Device(w, S.make_inputs(w))
    dev2.forward()
    torch.cuda.synchronize()
    first = N // 2 // C * C if what.startswith("future") else N // 3 // C * C
    if what != "leaf":
        assert torch.equal(dev.idx[:, :, :first], dev2.idx[:, :, :first])
        assert torch.equal(dev.lse[:, :, :first], dev2.lse[:, :, :first])
        _same(dev.out[:, :first], dev2.out[:, :first], (tensor, what))


def _check_backward(dev, idx, dout, got, C):
    """Which gradients must, may and must not be finite, and the finite ones against float64: the bound of check_gradient_rows
    with a tenth of the root mean square in place of its terms for the rounding of `out` inside delta (a wrong or a missing row
    is an error of the order of a whole gradient)."""
    B, N, Hq, d = dev.q.shape
    Hkv, G = dev.k.shape[2], Hq // dev.k.shape[2]
    leaf, t = torch.arange(N, device="cuda") // C, torch.arange(N, device="cuda")
    fin = lambda x: torch.isfinite(x).all(-1)  # noqa: E731
    dq, dk, dv = got
    ref = [torch.zeros(x.shape, dtype=torch.float64, device="cuda") for x in got]
    bad = [torch.zeros(x.shape[:3], dtype=torch.bool, device="cuda") for x in got]
    num = lambda x: torch.nan_to_num(x.double(), 0.0, 0.0, 0.0)  # noqa: E731
    for b in range(B):
        for h in range(Hkv):
            rows = idx[b, h].long()
            kept = torch.zeros((N, int(leaf[-1]) + 2), dtype=torch.bool, device="cuda").scatter_(1, torch.where(rows < 0, int(leaf[-1]) + 1, rows), True)
            see = kept[:, leaf] & (t[None, :] <= t[:, None])
            k, v = dev.k[b, :, h], dev.v[b, :, h]
            may_v = torch.zeros(N, dtype=torch.bool, device="cuda")
            for hq in range(h * G, h * G + G):
                has = see.any(1)
                bl = has & (~fin(dev.q[b, :, hq]) | (see & ~fin(k)[None]).any(1))
                bo = has & ~fin(dout[b, :, hq])
                ba = bl | bo | (has & (see & ~fin(v)[None]).any(1))
                bad[0][b, :, hq] = ba
                bad[1][b, :, h] |= (see & ba[:, None]).any(0)
                bad[2][b, :, h] |= (see & (bl | bo)[:, None]).any(0)
                may_v |= (see & ba[:, None]).any(0)
                good = (has & ~ba)[:, None]
                known = (has & ~bl & ~bo)[:, None]           # (a NaN value leaves the weights alone)
                s = (num(dev.q[b, :, hq]) @ num(k).T * d ** -0.5).masked_fill(~see, -math.inf)
                p = torch.where(known, torch.nan_to_num(torch.softmax(s, 1), 0.0), 0.0)
                do, o = num(dout[b, :, hq]), p @ num(v)
                ds = torch.where(good, p, 0.0) * (do @ num(v).T - (o * do).sum(1, keepdim=True)) * d ** -0.5
                ref[0][b, :, hq] = ds @ num(k)
                ref[1][b, :, h] += ds.T @ num(dev.q[b, :, hq])
                ref[2][b, :, h] += p.T @ do
            gone = ~fin(dv[b, :, h])
            assert bool((bad[2][b, :, h] <= gone).all()) and bool((gone <= may_v).all()), ("dv", b, h)
            bad[2][b, :, h] = gone
    assert torch.equal(~torch.isfinite(dq), bad[0][..., None].expand_as(dq)), "dq"
    assert torch.equal(~torch.isfinite(dk), bad[1][..., None].expand_as(dk)), "dk"
    for nm, x, r, m in zip(("dq", "dk", "dv"), got, ref, bad):
        x, r = torch.where(m[..., None], 0.0, x.double()), torch.where(m[..., None], 0.0, r)
        rms = float(r.square().mean().sqrt())
        err, bound = (x - r).abs(), 2.0 ** -5 * r.abs().amax(-1, keepdim=True) + 0.1 * rms
        assert bool((err <= bound).all()), (nm, float((err - bound).max()), rms)


# uniform batches: every group size and block size, one and two tiles per item, split and unsplit key blocks
BACKWARD = [(1, 700, 8, 2, 128, 64, 2, 4), (2, 500, 4, 1, 64, 128, 2, 3), (1, 1100, 2, 2, 64, 64, 2, 5), (1, 450, 16, 1, 128, 64, 4, 3),
            (3, 900, 32, 8, 64, 128, 2, 3)]


@pytest.mark.parametrize("shape", BACKWARD, ids=lambda s: "b%d_n%d_h%d_%d_d%d_c%d_g%d_k%d" % s)
@pytest.mark.parametrize("tensor", ["q", "k", "v", "dout"])
@pytest.mark.parametrize("what", ["future", "key", "leaf"])
def test_dense_backward_shows_what_its_rows_selected(shape, tensor, what):
    B, N, Hq, Hkv, d, C, g, K = shape
    w = S.Workload("nf_bwd", B, N, Hq, Hkv, d, C, g, K, "bf16", 2500 + N, "iid")
    dev = T.Device(w, S.make_inputs(w))
    dout = torch.randn(dev.q.shape, generator=torch.Generator(device="cuda").manual_seed(4), device="cuda").bfloat16()
    x = dout if tensor == "dout" else getattr(dev, tensor)
    if what == "future":
        x[:, N // 2 + 9:] = NAN
    elif what == "key":
        x[:, N // 3, 0, 5] = NAN
        x[:, N // 3 + C, -1, 7] = math.inf if tensor in ("v", "dout") else NAN
    else:
        x[-1, N // 3 // C * C:N // 3 // C * C + C] = NAN
    dev.forward()
    assert dev.sync_status() == 0
    got = [torch.full_like(y, 7.0) for y in (dev.q, dev.k, dev.v)]
    ws = PB.alloc_workspace(dev.p, PB.OP_BSA_BWD)
    P.pisa_bsa_bwd(dev.p, dev.q, dev.k, dev.v, dev.idx, dev.out, dev.lse, dout, *got, ws)
    torch.cuda.synchronize()
    assert P.read_status(ws) == 0
    _check_backward(dev, dev.idx, dout, got, C)


@pytest.mark.parametrize("shape", BACKWARD[:3], ids=lambda s: "b%d_n%d_h%d_%d_d%d_c%d_g%d_k%d" % s)
def test_padded_rows_without_blocks_reach_no_gradient(shape):
    """Rows whose blocks were set to -1 may hold anything: queries, gradients, outputs and denominators."""
    B, N, Hq, Hkv, d, C, g, K = shape
    w = S.Workload("nf_pad", B, N, Hq, Hkv, d, C, g, K, "bf16", 2600 + N, "iid")
    dev = T.Device(w, S.make_inputs(w))
    dev.forward()
    assert dev.sync_status() == 0
    dout = torch.randn(dev.q.shape, generator=torch.Generator(device="cuda").manual_seed(4), device="cuda").bfloat16()
    end = N - 2 * C - 37                                    # inside a leaf and a tile
    idx = dev.idx.clone()
    idx[:, :, end:] = -1
    for x in (dev.q, dout, dev.out):
        x[:, end:] = NAN
    for x in (dev.k, dev.v):
        x[:, end:] = math.inf
    for fill in (0.0, NAN, math.inf):
        dev.lse[:, :, end:] = fill
        got = [torch.full_like(y, 7.0) for y in (dev.q, dev.k, dev.v)]
        ws = PB.alloc_workspace(dev.p, PB.OP_BSA_BWD)
        P.pisa_bsa_bwd(dev.p, dev.q, dev.k, dev.v, idx, dev.out, dev.lse, dout, *got, ws)
        torch.cuda.synchronize()
        assert P.read_status(ws) == 0
        _check_backward(dev, idx, dout, got, C)
        for x in got:
            assert bool((x[:, end:] == 0).all()), fill
