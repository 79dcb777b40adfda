"""The dense masked backward at the sizes where it can go wrong (tile and step edges, split key items, one and two tiles per
item, packed neighbours), on both outcomes of the choice that the rows make on the device for longer sequences, and with
rows and key blocks nobody selected.  Bounds: those of test_gpu_backward."""
import numpy as np
import pytest
import torch

import pisa_synth as S
from oracle import pisa_oracle as O

pytestmark = pytest.mark.gpu

import pisa_testlib as T  # noqa: E402
import paper_2609_31093_b200 as P  # noqa: E402
from paper_2609_31093_b200 import binding as PB  # noqa: E402

CASES = [
    # B, N, Hq, Hkv, d, C, g, K, queries repeated over this many tokens
    (1, 127, 4, 1, 128, 64, 2, 3, 1), (1, 129, 2, 2, 64, 128, 2, 3, 1), (2, 257, 1, 1, 128, 128, 2, 3, 1),
    (1, 1000, 16, 1, 64, 64, 2, 4, 1), (1, 1152, 8, 2, 128, 128, 2, 3, 1),
    (1, 1153, 8, 2, 128, 128, 2, 3, 1), (1, 2500, 4, 1, 128, 64, 2, 4, 1),        # the rows decide: lists
    (1, 2500, 4, 1, 128, 64, 2, 4, 128), (1, 3000, 8, 2, 64, 128, 2, 4, 200),     # ... dense
    (3, 1500, 16, 8, 128, 64, 4, 4, 1),                                           # two tiles per item, no split
]


def _dk_rounding(dev, dout, w):
    """What the bf16 roundings of dS (2^-9 of each) and of `out` inside delta = dO . O do to dK = sum dS_i q_i: six standard
    deviations of independent roundings, each uniform in its interval.  Rows that share one query add multiples of a single
    vector, so where their dS cancel a whole row of dK is small and a bound relative to its maximum says nothing."""
    u = 2.0 ** -9 / 3 ** 0.5
    G, scale = w.Hq // w.Hkv, w.d ** -0.5
    extra = torch.zeros(dev.k.shape, dtype=torch.float64, device="cuda")
    key_leaf = torch.arange(w.N, device="cuda") // w.C
    causal = torch.arange(w.N, device="cuda")[None, :] <= torch.arange(w.N, device="cuda")[:, None]
    for b in range(w.B):
        for h in range(w.Hkv):
            k, v = dev.k[b, :, h].double(), dev.v[b, :, h].double()
            rows = dev.idx[b, h].long()
            kept = torch.zeros((w.N, int(key_leaf[-1]) + 2), dtype=torch.bool, device="cuda").scatter_(1, torch.where(rows < 0, int(key_leaf[-1]) + 1, rows), True)
            see = kept[:, key_leaf] & causal
            for hq in range(h * G, (h + 1) * G):
                q, do, o = dev.q[b, :, hq].double(), dout[b, :, hq].double(), dev.out[b, :, hq].double()
                p = torch.softmax((q @ k.T * scale).masked_fill(~see, float("-inf")), dim=1)
                ds = p * (do @ v.T - (o * do).sum(1, keepdim=True)) * scale
                var = ds.square() + (p * scale).square() * (o * do).square().sum(1, keepdim=True)
                extra[b, :, h] += var.T @ q.square()
    return 6 * u * extra.sqrt().cpu().numpy()


def _check(name, t, idx, out, dout_bits, got, w, dk_extra=0.0):
    rq, rk, rv = O.attend_backward(t["q"], t["k"], t["v"], idx.cpu().numpy(), dout_bits, C=w.C, dtype="bf16")
    o64 = out.to(torch.float64).cpu().numpy()
    do64 = O.load_storage(dout_bits, "bf16")
    kmax = float(np.abs(O.load_storage(t["k"], "bf16")).max())
    d_delta = 2.0 ** -9 * np.abs(o64 * do64).sum(axis=-1, keepdims=True) / np.sqrt(w.d) * kmax
    for nm, g, ref, extra in (("dq", got[0], rq, d_delta), ("dk", got[1], rk, dk_extra), ("dv", got[2], rv, 0.0)):
        g64 = g.to(torch.float64).cpu().numpy()
        assert np.isfinite(g64).all(), (name, nm)
        T.check_gradient_rows(f"{name}.{nm}", g64, ref, extra)


@pytest.mark.parametrize("shape", CASES, ids=lambda s: "b%d_n%d_h%d_%d_d%d_c%d_g%d_k%d_r%d" % s)
def test_gradients_match_the_oracle(shape):
    B, N, Hq, Hkv, d, C, g, K, rep = shape
    w = S.Workload("bwdd", B, N, Hq, Hkv, d, C, g, K, "bf16", 640 + N % 97, "iid")
    t = S.make_inputs(w)
    if rep > 1:
        t["q"] = np.ascontiguousarray(t["q"][:, (np.arange(N) // rep) * rep])
    dev = T.Device(w, t)
    dev.forward()
    assert dev.sync_status() == 0
    rng = np.random.default_rng(w.seed)
    dout_bits = S.f32_to_bf16_bits(rng.standard_normal(t["q"].shape).astype(np.float32))
    got = [torch.full_like(x, float("nan")) for x in (dev.q, dev.k, dev.v)]
    ws = PB.alloc_workspace(dev.p, PB.OP_BSA_BWD)
    for _ in range(2):
        P.pisa_bsa_bwd(dev.p, dev.q, dev.k, dev.v, dev.idx, dev.out, dev.lse, T.to_torch(dout_bits, "bf16"), *got, ws)
    torch.cuda.synchronize()
    assert P.read_status(ws) == 0
    _check("n%d" % N, t, dev.idx, dev.out, dout_bits, got, w,
           _dk_rounding(dev, T.to_torch(dout_bits, "bf16"), w) if rep > 1 else 0.0)


def test_rows_without_blocks_and_blocks_without_rows_get_zeros():
    """idx rows of -1 only (denominator -inf) have no gradient and add none; key blocks nobody selected get zeros."""
    w = S.Workload("bwdz", 1, 700, 8, 2, 128, 64, 2, 4, "bf16", 655, "iid")
    t = S.make_inputs(w)
    dev = T.Device(w, t)
    dev.forward()
    idx = dev.idx.clone()
    idx[:, :, 64:192] = -1                                  # whole tiles without a block
    idx[:, :, 300] = -1
    idx[idx == 5] = -1                                      # nobody selects keys 320 .. 383
    P.pisa_bsa_fwd(dev.p, dev.q, dev.k, dev.v, idx, dev.out, dev.lse, dev.ws)
    dout = torch.randn_like(dev.q)
    dq, dk, dv = (torch.full_like(x, float("nan")) for x in (dev.q, dev.k, dev.v))
    ws = PB.alloc_workspace(dev.p, PB.OP_BSA_BWD)
    P.pisa_bsa_bwd(dev.p, dev.q, dev.k, dev.v, idx, dev.out, dev.lse, dout, dq, dk, dv, ws)
    torch.cuda.synchronize()
    assert P.read_status(ws) == 0
    assert all(bool(torch.isfinite(x).all()) for x in (dq, dk, dv))
    assert bool((dq[:, 64:192] == 0).all()) and bool((dq[:, 300] == 0).all())
    assert bool((dk[:, 320:384] == 0).all()) and bool((dv[:, 320:384] == 0).all())
    assert float(dk[:, :64].float().abs().max()) > 0


def test_packed_gradients_do_not_see_the_neighbours():
    """Whatever lies in a neighbouring sequence, NaN and infinities included, must not reach a gradient."""
    lens = [127, 1, 128, 129, 255, 64, 1000, 63, 31, 640]
    Hq, Hkv, d, C, g, K = 8, 2, 128, 64, 2, 4
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    total = int(cu[-1])
    w = S.Workload("bwdn", 1, total, Hq, Hkv, d, C, g, K, "bf16", 660, "iid")
    t = S.make_inputs(w)
    q, k, v = (T.to_torch(t[x][0], "bf16") for x in ("q", "k", "v"))
    dout = torch.randn_like(q)
    p = P.Params(1, max(lens), Hq, Hkv, d, C, g, K, dtype="bf16")
    pyramid, ws, wsb = PB.alloc_pyramid(p), PB.alloc_workspace(p, PB.OP_FORWARD_PACKED), PB.alloc_workspace(p, PB.OP_BSA_BWD_PACKED)
    idx = torch.zeros((Hkv * K * total,), dtype=torch.int32, device="cuda")
    out, lse = torch.zeros_like(q), torch.zeros((Hq * total,), dtype=torch.float32, device="cuda")
    P.pisa_forward_packed(p, cu.tolist(), q, k, v, pyramid, idx, out, lse, ws)

    def run():
        got = [torch.full_like(x, float("nan")) for x in (q, k, v)]
        P.pisa_bsa_bwd_packed(p, cu.tolist(), q, k, v, idx, out, lse, dout, *got, wsb)
        torch.cuda.synchronize()
        assert P.read_status(wsb) == 0
        return got

    clean = run()
    for i in range(1, len(lens), 2):
        for x in (q, k, v, out, dout):
            x[cu[i]:cu[i + 1]] = float("nan")
            x[cu[i]:cu[i] + 1] = float("inf")
    dirty = run()
    for i in range(0, len(lens), 2):
        a, b = int(cu[i]), int(cu[i + 1])
        for x, y in zip(clean, dirty):
            assert bool(torch.isfinite(y[a:b]).all()), i
            # (split key items add their parts in any order: fp32 rounding, one bf16 step at most)
            assert torch.allclose(x[a:b].float(), y[a:b].float(), rtol=2.0 ** -7, atol=1e-5), i
