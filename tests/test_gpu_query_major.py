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
