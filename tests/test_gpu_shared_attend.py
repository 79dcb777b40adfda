"""Attention of the list-driven forward: leaves that a query tile's rows share are served query-major, the others by the lists.
Every group size, leaf size and head dimension, lengths that end inside a tile, lists of an odd number of 64-key leaves."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu

import paper_2609_31093_b200 as P  # noqa: E402
from paper_2609_31093_b200 import binding as PB  # noqa: E402

SHAPES = [
    # N, Hq, Hkv, d, C, g, K: longer than what the dense kernels take
    (3111, 8, 2, 128, 64, 2, 3), (3073, 8, 2, 64, 64, 4, 3), (6181, 2, 2, 128, 64, 2, 3), (6145, 2, 2, 64, 128, 2, 3),
    (3099, 16, 1, 64, 64, 2, 3), (2819, 4, 2, 128, 128, 2, 4), (3200, 16, 2, 128, 64, 4, 3), (8225, 8, 2, 128, 64, 2, 8),
    (5700, 4, 1, 128, 128, 2, 8),
]


def _tensors(N, Hq, Hkv, d, seed):
    """Passages of some 200 tokens on a few topics: neighbouring queries find the same blocks, others find others."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    normal = lambda *s: torch.randn(s, generator=gen, device="cuda")  # noqa: E731
    which = torch.randint(0, 6, (N + 1,), generator=gen, device="cuda")[(torch.rand(N, generator=gen, device="cuda") < 1 / 200).cumsum(0)]
    mean = 0.6 * normal(6, d)[which]
    q = (normal(1, N, Hq, d) + mean[None, :, None]).bfloat16()
    k = (normal(1, N, Hkv, d) + mean[None, :, None]).bfloat16()
    return q, k, normal(1, N, Hkv, d).bfloat16()


def _forward(shape, q, k, v):
    N, Hq, Hkv, d, C, g, K = shape
    p = P.Params(1, N, Hq, Hkv, d, C, g, K)
    idx = torch.full((1, Hkv, N, K), -7, dtype=torch.int32, device="cuda")
    out, lse = torch.full_like(q, 7.0), torch.zeros((1, Hq, N), dtype=torch.float32, device="cuda")
    ws = PB.alloc_workspace(p, PB.OP_FORWARD)
    ws.fill_(0x5a)                                    # nothing may rest on a cleared workspace
    P.set_stage_timing(True)
    P.set_forward_chunks(1)
    try:
        P.pisa_forward(p, q, k, v, PB.alloc_pyramid(p), idx, out, lse, ws)
        torch.cuda.synchronize()
        assert "shared_attend" in P.get_kernel_ms()
    finally:
        P.set_stage_timing(False)
        P.set_forward_chunks(0)
    assert P.read_status(ws) == 0
    return idx, out, lse


def _kept(idx, N, C, h):
    leaf = torch.arange(N, device="cuda") // C
    rows = idx[0, h].long()
    n = int(leaf[-1]) + 2
    return torch.zeros((N, n), dtype=torch.bool, device="cuda").scatter_(1, torch.where(rows < 0, n - 1, rows), True)


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "n%d_h%d_%d_d%d_c%d_g%d_k%d" % s)
def test_shared_and_listed_leaves_make_up_the_attention(shape):
    N, Hq, Hkv, d, C, g, K = shape
    q, k, v = _tensors(N, Hq, Hkv, d, 31 + N)
    idx, out, lse = _forward(shape, q, k, v)
    t, G = torch.arange(N, device="cuda"), Hq // Hkv
    shared = listed = 0
    for h in range(Hkv):
        kept = _kept(idx, N, C, h)
        tile = kept[:, :-1].float().split(128 // G)
        shared += sum(int((x.mean(0) >= 0.5).sum()) for x in tile)
        listed += sum(int(((x.mean(0) > 0) & (x.mean(0) < 0.1)).sum()) for x in tile)
        see = kept[:, t // C] & (t[None] <= t[:, None])
        for hq in range(h * G, (h + 1) * G):
            s = (q[0, :, hq].double() @ k[0, :, h].double().T / math.sqrt(d)).masked_fill(~see, -math.inf)
            # the bounds of the bf16 outputs everywhere in these tests: both sides round to 8 bits, values below 2.56
            err = (out[0, :, hq].double() - torch.softmax(s, 1) @ v[0, :, h].double()).abs()
            big = v.abs().max().double() > 2.56
            assert float(err.max()) <= 2e-2 + (2 ** -7 * float(out.abs().max()) if big else 0) and float(err.mean()) <= 2e-3
            assert float((lse[0, hq].double() - torch.logsumexp(s, 1)).abs().max()) <= 1e-4
    assert shared > 0 and (listed > 0 or K == 3)


@pytest.mark.parametrize("shape", [SHAPES[i] for i in (0, 2, 3, 4, 7)], ids=lambda s: "n%d_h%d_%d_d%d_c%d_g%d_k%d" % s)
def test_a_value_that_is_not_finite_reaches_only_rows_that_selected_it(shape):
    N, Hq, Hkv, d, C, g, K = shape
    q, k, v = _tensors(N, Hq, Hkv, d, 57 + N)
    idx, clean, _ = _forward(shape, q, k, v)
    G = Hq // Hkv
    leaf = N // C // 2
    for bad in (math.nan, math.inf):
        x = v.clone()
        x[0, leaf * C + 5, :, ::3] = bad
        idx2, out, _ = _forward(shape, q, k, x)
        assert torch.equal(idx, idx2)
        for h in range(Hkv):
            has = _kept(idx, N, C, h)[:, leaf]
            rows = out[0, :, h * G:(h + 1) * G].float()
            assert torch.isfinite(rows[~has]).all()
            # (fp32 additions into the accumulator come in any order, the recomputed rows sum in another one)
            assert float((rows - clean[0, :, h * G:(h + 1) * G].float())[~has].abs().max()) <= 2 ** -7 * max(1.0, float(clean.abs().max()))
            after = has & (torch.arange(N, device="cuda") >= (leaf + 1) * C)
            assert not torch.isfinite(rows[after][:, :, ::3]).any()


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "n%d_h%d_%d_d%d_c%d_g%d_k%d" % s)
def test_leaf_scores_of_shared_and_listed_nodes(shape):
    """The routing's per-leaf denominators (whichever kernel scored the leaf, in whichever place of the row) against float64:
    2e-6 relative for ex2.approx and the sums of up to 128 terms, 2^-22 of the logits' size for their fp32 accumulation."""
    N, Hq, Hkv, d, C, g, K = shape
    q, k, _ = _tensors(N, Hq, Hkv, d, 91 + N)
    p = P.Params(1, N, Hq, Hkv, d, C, g, K)
    pyramid, ws = PB.alloc_pyramid(p), PB.alloc_workspace(p, PB.OP_ROUTE)
    ws.fill_(0x5a)
    P.pisa_build_pyramid(p, k, pyramid)
    idx = torch.full((1, Hkv, N, K), -7, dtype=torch.int32, device="cuda")
    sel = torch.full((1, Hq, N, K), 7.0, dtype=torch.float32, device="cuda")
    P.pisa_route(p, q, k, pyramid, idx, None, ws, sel_lse=sel)
    torch.cuda.synchronize()
    assert P.read_status(ws) == 0
    t, G = torch.arange(N, device="cuda"), Hq // Hkv
    M1 = (N + C - 1) // C
    for h in range(Hkv):
        rows = idx[0, h].long()
        for hq in range(h * G, (h + 1) * G):
            s = (q[0, :, hq].double() @ k[0, :, h].double().T / math.sqrt(d)).masked_fill(t[None] > t[:, None], -math.inf)
            s = torch.nn.functional.pad(s, (0, M1 * C - N), value=-math.inf).view(N, M1, C)
            ref = torch.logsumexp(s, 2).gather(1, rows.clamp(min=0))
            got = sel[0, hq].double()
            assert bool((got[rows < 0] == -math.inf).all())
            assert float((got - ref).abs()[rows >= 0].max()) <= 2e-6 + 2 ** -22 * float(s[s > -math.inf].abs().max())
