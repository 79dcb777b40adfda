"""The decoding kernel's branches: up-front and level-by-level scoring, one and two warps per leaf, every group size's
instantiation, fan-ins beside two, and the cluster widths down to two CTAs per SM in more than one wave."""
import pytest
import torch

import pisa_synth as S

pytestmark = pytest.mark.gpu

import pisa_testlib as T  # noqa: E402
import test_gpu_decode as D  # noqa: E402
import paper_2609_31093_b200 as P  # noqa: E402
from paper_2609_31093_b200 import binding as PB  # noqa: E402

CASES = [
    # B, N, Hq, Hkv, d, C, g, K
    (1, 270000, 2, 1, 64, 32, 2, 4),      # more than 4096 live nodes above the leaves: scored level by level
    (1, 6000, 16, 1, 128, 128, 2, 32),    # G = 16, 64 candidates
    (1, 2600, 8, 1, 64, 64, 4, 32),       # G = 8, 128 candidates, fan-in 4
    (2, 1500, 4, 2, 128, 64, 3, 5),       # fan-in 3
    (3, 2500, 8, 8, 64, 64, 4, 8),        # G = 1
    (40, 700, 8, 4, 128, 64, 2, 4),       # 160 units: two CTAs per SM, more than one wave
]


@pytest.mark.parametrize("shape", CASES, ids=lambda s: "b%d_n%d_h%d_%d_d%d_c%d_g%d_k%d" % s)
def test_steps_match_the_oracle(shape):
    B, N, Hq, Hkv, d, C, g, K = shape
    w = S.Workload("decb", B, N, Hq, Hkv, d, C, g, K, "bf16", 430 + K, "iid")
    t = S.make_inputs(w)
    n0 = N - 3
    cache = D.Cache(w, t, cap=N, filled=n0)
    P.pisa_build_pyramid(cache.p, cache.k, cache.pyr)
    for pos in range(n0, N):
        cache.step(pos)
        if pos != n0 + 1:
            D._check_step(cache, t, pos)
    # the path of the last token, against the pyramid built from the whole sequence (at most one bf16 ulp off)
    ref = torch.empty_like(cache.pyr)
    P.pisa_build_pyramid(cache.p, cache.k, ref)
    for l in range(1, cache.L + 1):
        n = B * Hkv * cache.M[l] * d
        want = ref[cache.off[l]:cache.off[l] + n].view(B, Hkv, cache.M[l], d)[:, :, -1].float()
        got = cache.level(l)[:, :, -1].float()
        assert bool(((got - want).abs() <= 2.0 ** -7 * want.abs() + 1e-6).all()), l


@pytest.mark.parametrize("units", [61681, 65535])          # units and refreshing clusters: more than 65535 clusters
def test_as_many_sequences_as_the_library_takes(units):
    N, d, C, pos = 64, 64, 32, 40
    gen = torch.Generator(device="cuda").manual_seed(3)
    q, k, v = (torch.randn(s, generator=gen, device="cuda").bfloat16() for s in ((units, 1, d), (units, N, 1, d), (units, N, 1, d)))
    p = P.Params(units, N, 1, 1, d, C, 2, 3, dtype="bf16")
    pyr = PB.alloc_pyramid(p)
    pyr.fill_(float("nan"))
    P.pisa_build_pyramid(p, k, pyr)
    L, M, off, _ = P.pyramid_layout(p)
    idx = torch.full((units, 1, 3), -7, dtype=torch.int32, device="cuda")
    out, lse, ws = torch.zeros_like(q), torch.zeros((units, 1), device="cuda"), PB.alloc_workspace(p, PB.OP_DECODE)
    P.pisa_decode_step(p, pos, q, k, v, pyr, idx, out, lse, ws)
    torch.cuda.synchronize()
    assert P.read_status(ws) == 0
    assert bool((idx == torch.tensor([0, 1, -1], device="cuda", dtype=torch.int32)).all())
    z = torch.einsum("bd,bnd->bn", q[:, 0].float(), k[:, :pos + 1, 0].float()) * d ** -0.5
    assert torch.allclose(lse[:, 0], torch.logsumexp(z, 1), rtol=1e-4, atol=1e-4)
    want = torch.einsum("bn,bnd->bd", torch.softmax(z, 1), v[:, :pos + 1, 0].float())
    assert float((out[:, 0].float() - want).abs().max()) <= T.BF16_MAX_ABS
    for l in range(1, L + 1):                               # the path: leaf 1 holds nine keys so far
        node = pyr[off[l]:off[l] + units * M[l] * d].view(units, M[l], d)[:, -1].float()
        leaf1 = k[:, C:pos + 1, 0].float().mean(1)
        ref = leaf1 if l == 1 else (k[:, :C, 0].float().mean(1) + leaf1) / 2
        assert float((node - ref).abs().max()) <= 2.0 ** -7 * 2
