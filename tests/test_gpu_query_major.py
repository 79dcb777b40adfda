"""The query-major path (dense scoring, one-thread-per-token selection, masked dense attention) at the sizes where it can
go wrong: lengths around its tiles (128 / G tokens, 256 / G with two tiles per item), its 128-key steps, the first level
that prunes, its longest sequences, and one token past them (where the list-driven path takes over)."""
import numpy as np
import pytest

import pisa_synth as S

pytestmark = pytest.mark.gpu

import pisa_testlib as T  # noqa: E402

CASES = [
    # B, N, Hq, Hkv, d, C, g, K
    (1, 127, 4, 1, 128, 64, 2, 3), (1, 128, 4, 1, 64, 64, 2, 3), (1, 129, 4, 1, 128, 128, 2, 3),
    (1, 5 * 64, 2, 2, 128, 64, 2, 4), (1, 5 * 64 + 1, 2, 2, 64, 64, 4, 4),          # M1 = K + 1: only the leaf level prunes
    (2, 1023, 16, 1, 64, 64, 2, 5), (2, 1025, 1, 1, 128, 128, 4, 5),                # G = 16: 8 tokens per tile; G = 1: 128
    (3, 2049, 8, 4, 128, 64, 4, 7), (1, 3583, 16, 2, 128, 64, 2, 12),               # G = 2 and 8, ragged levels
    (1, 3 * 704, 8, 2, 64, 128, 2, 3), (1, 3 * 704 + 1, 8, 2, 64, 128, 2, 3),       # the longest dense sequence, and one more token
    (4, 5000, 32, 8, 64, 64, 4, 32),                                                # g * K = 128 candidates, two tiles per item
    (1, 9001, 16, 16, 128, 64, 2, 16),                                              # two tiles per item, G = 1
]


@pytest.mark.parametrize("shape", CASES, ids=lambda s: "b%d_n%d_h%d_%d_d%d_c%d_g%d_k%d" % s)
def test_forward_matches_the_oracle(shape):
    B, N, Hq, Hkv, d, C, g, K = shape
    w = S.Workload("qm", B, N, Hq, Hkv, d, C, g, K, "bf16", 1700 + N, "iid")
    t = S.make_inputs(w)
    dev = T.Device(w, t)
    dev.forward()
    assert dev.sync_status() == 0
    tri = S.sample_queries(w, 24, B=B)
    last = np.array([[b, h, p] for b in range(B) for h in range(Hkv) for p in {N - 1, max(N - 2, 0), 0}])
    T.check_forward_dev(dev, T.oracle_problem(w, t), np.concatenate([tri, last]))


def test_packed_sequences_do_not_see_their_neighbours():
    """Packed sequences share the TMA tiles of their last keys with the next sequence: whatever lies there, NaN and
    infinities included, must not reach a row.  Lengths around tile and step edges, one set of launches for all."""
    import torch
    import paper_2609_31093_b200 as P
    from paper_2609_31093_b200 import binding as PB
    lens = [127, 1, 128, 129, 255, 64, 1000, 63, 31, 640]
    Hq, Hkv, d, C, g, K = 8, 2, 128, 64, 2, 4
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    total = int(cu[-1])
    w = S.Workload("qm_nan", 1, total, Hq, Hkv, d, C, g, K, "bf16", 1790, "iid")
    t = S.make_inputs(w)
    q, k, v = (T.to_torch(t[x][0], "bf16") for x in ("q", "k", "v"))
    p = P.Params(1, max(lens), Hq, Hkv, d, C, g, K, dtype="bf16")
    pyramid, ws = PB.alloc_pyramid(p), PB.alloc_workspace(p, PB.OP_FORWARD_PACKED)

    def run():
        idx = torch.full((Hkv * K * total,), -7, dtype=torch.int32, device="cuda")
        out, lse = torch.zeros_like(q), torch.zeros((Hq * total,), dtype=torch.float32, device="cuda")
        P.pisa_forward_packed(p, cu.tolist(), q, k, v, pyramid, idx, out, lse, ws)
        torch.cuda.synchronize()
        assert P.read_status(ws) == 0
        return idx, out, lse

    clean = run()
    for i in range(1, len(lens), 2):                       # every second sequence turns into NaN and infinity
        for x in (q, k, v):
            x[cu[i]:cu[i + 1]] = float("nan")
            x[cu[i]:cu[i] + 1] = float("inf")
    dirty = run()
    for i in range(0, len(lens), 2):
        a, b = int(cu[i]), int(cu[i + 1])
        assert torch.equal(dirty[0][Hkv * K * a:Hkv * K * b], clean[0][Hkv * K * a:Hkv * K * b]), i
        assert torch.equal(dirty[1][a:b], clean[1][a:b]), i
        assert torch.equal(dirty[2][Hq * a:Hq * b], clean[2][Hq * a:Hq * b]), i


@pytest.mark.parametrize("shape", [(1, 3000, 32, 8, 128, 128, 4, 5), (2, 1500, 4, 4, 64, 128, 4, 3), (1, 60, 8, 2, 128, 64, 2, 4)],
                         ids=lambda s: "b%d_n%d_h%d_%d_d%d_c%d_g%d_k%d" % s)
@pytest.mark.parametrize("packed", [False, True])
def test_shapes_without_lists_keep_the_exact_paths_precision(shape, packed):
    """Shapes that the list-driven kernels do not take (fan-in 4 with C = 128; one leaf) ran on the exact fp32 path, which does
    not round the probabilities: the dense kernels are no further from float64 (the rounding of the output, 2^-9, dominates;
    one bf16 term per probability adds a quarter to the error)."""
    import torch
    import paper_2609_31093_b200 as P
    from paper_2609_31093_b200 import binding as PB
    B, N, Hq, Hkv, d, C, g, K = shape
    w = S.Workload("qm_prec", B, N, Hq, Hkv, d, C, g, K, "bf16", 1795 + N, "iid")
    dev = T.Device(w, S.make_inputs(w))
    dev.forward()
    if packed:
        cu = [N * b for b in range(B + 1)]
        p = P.Params(1, N, Hq, Hkv, d, C, g, K, dtype="bf16")
        ws = PB.alloc_workspace(p, PB.OP_FORWARD_PACKED)
        P.pisa_forward_packed(p, cu, dev.q, dev.k, dev.v, PB.alloc_pyramid(p), dev.idx, dev.out, dev.lse, ws)
    assert dev.sync_status() == 0
    ref = T.Device(w, S.make_inputs(w), impl=PB.IMPL_SIMT)
    ref.bsa(dev.idx)
    assert ref.sync_status() == 0
    leaf, t = torch.arange(N, device="cuda") // C, torch.arange(N, device="cuda")
    err = [0.0, 0.0]
    for b in range(B):
        for h in range(Hkv):
            rows = dev.idx[b, h].long()
            kept = torch.zeros((N, int(leaf[-1]) + 2), dtype=torch.bool, device="cuda").scatter_(1, torch.where(rows < 0, int(leaf[-1]) + 1, rows), True)
            see = kept[:, leaf] & (t[None] <= t[:, None])
            for hq in range(h * Hq // Hkv, (h + 1) * Hq // Hkv):
                s = (dev.q[b, :, hq].double() @ dev.k[b, :, h].double().T * d ** -0.5).masked_fill(~see, float("-inf"))
                o = torch.softmax(s, 1) @ dev.v[b, :, h].double()
                for i, x in enumerate((dev.out, ref.out)):
                    err[i] += float((x[b, :, hq].double() - o).square().sum())
    err = [e ** 0.5 for e in err]
    print("dense %.6e exact path %.6e ratio %.4f" % (err[0], err[1], err[0] / err[1]))
    assert err[0] <= 1.002 * err[1]
