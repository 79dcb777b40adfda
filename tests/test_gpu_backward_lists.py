"""The list-driven backward: every group size (how the reductions are made 16 bytes wide depends on it), leaf size and head
dimension, at lengths past those that the dense kernels always take, with queries that share nothing, so that the lists run."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu

import pisa_testlib as T  # noqa: E402
import paper_2609_31093_b200 as P  # noqa: E402
from paper_2609_31093_b200 import binding as PB  # noqa: E402

SHAPES = [
    # B, N, Hq, Hkv, d, C, g, K
    (1, 1501, 2, 2, 128, 64, 2, 3), (1, 1030, 2, 1, 128, 64, 2, 3), (1, 900, 4, 2, 64, 128, 2, 3), (2, 1000, 8, 2, 128, 64, 4, 3),
    (1, 777, 8, 2, 128, 128, 2, 3), (1, 2100, 8, 1, 64, 64, 2, 3), (1, 1700, 16, 1, 128, 64, 2, 3), (1, 1400, 2, 2, 64, 128, 2, 3),
]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "b%d_n%d_h%d_%d_d%d_c%d_g%d_k%d" % s)
def test_gradients_of_listed_blocks(shape):
    B, N, Hq, Hkv, d, C, g, K = shape
    gen = torch.Generator(device="cuda").manual_seed(71 + N)
    q, k, v, dout = (torch.randn((B, N, h, d), generator=gen, device="cuda").bfloat16() for h in (Hq, Hkv, Hkv, Hq))
    p = P.Params(B, N, Hq, Hkv, d, C, g, K)
    idx = torch.zeros((B, Hkv, N, K), dtype=torch.int32, device="cuda")
    out, lse = torch.zeros_like(q), torch.zeros((B, Hq, N), dtype=torch.float32, device="cuda")
    P.pisa_forward(p, q, k, v, PB.alloc_pyramid(p), idx, out, lse, PB.alloc_workspace(p, PB.OP_FORWARD))
    ws = PB.alloc_workspace(p, PB.OP_BSA_BWD)
    ws.fill_(0x5a)                                   # nothing may rest on a cleared workspace
    got = [torch.full_like(x, math.nan) for x in (q, k, v)]
    for _ in range(2):
        P.pisa_bsa_bwd(p, q, k, v, idx, out, lse, dout, *got, ws)
    torch.cuda.synchronize()
    assert P.read_status(ws) == 0
    leaf, t, G = torch.arange(N, device="cuda") // C, torch.arange(N, device="cuda"), Hq // Hkv
    ref = [torch.zeros(x.shape, dtype=torch.float64, device="cuda") for x in got]
    for b in range(B):
        for h in range(Hkv):
            rows = idx[b, h].long()
            n = int(leaf[-1]) + 2
            see = torch.zeros((N, n), dtype=torch.bool, device="cuda").scatter_(1, torch.where(rows < 0, n - 1, rows), True)[:, leaf]
            see &= t[None] <= t[:, None]
            for hq in range(h * G, h * G + G):
                s = (q[b, :, hq].double() @ k[b, :, h].double().T / math.sqrt(d)).masked_fill(~see, -math.inf)
                w, do = torch.softmax(s, 1), dout[b, :, hq].double()
                # (delta from the stored output, as the kernels take it)
                ds = w * (do @ v[b, :, h].double().T - (do * out[b, :, hq].double()).sum(1, keepdim=True)) / math.sqrt(d)
                ref[0][b, :, hq] = ds @ k[b, :, h].double()
                ref[1][b, :, h] += ds.T @ q[b, :, hq].double()
                ref[2][b, :, h] += w.T @ do
    for name, x, r in zip(("dq", "dk", "dv"), got, ref):
        T.check_gradient_rows(name, x.double().cpu().numpy(), r.cpu().numpy())
