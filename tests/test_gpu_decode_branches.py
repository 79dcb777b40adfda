"""The decoding kernel's branches: up-front and level-by-level scoring, one and two warps per leaf, every group size's
instantiation, fan-ins beside two, and the cluster widths down to two CTAs per SM in more than one wave."""
import pytest
import torch

import pisa_synth as S

pytestmark = pytest.mark.gpu

import test_gpu_decode as D  # noqa: E402
import paper_2609_31093_b200 as P  # noqa: E402

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
