"""The exact fp32 path at the row counts where a token's share of warps changes (eight, four, one), for every number of lanes
per key row and for groups of one and two.  Bounds: those of test_gpu_parity."""
import numpy as np
import pytest
import torch

import pisa_synth as S

pytestmark = pytest.mark.gpu

import pisa_testlib as T  # noqa: E402


def _cases():
    sms = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 148
    lo, hi = 5 * sms, 16 * sms
    return [(1, lo, 1, 1, 64, "fp32"), (1, lo + 1, 1, 1, 128, "fp32"), (1, hi, 2, 1, 32, "fp32"), (1, hi + 1, 1, 1, 64, "fp32"),
            (3, lo // 6, 4, 2, 64, "fp32"), (1, 65, 1, 1, 32, "fp32")]


@pytest.mark.parametrize("case", _cases(), ids=lambda c: "b%d_n%d_h%d_%d_d%d_%s" % c)
def test_forward_matches_the_oracle(case):
    B, N, Hq, Hkv, d, dtype = case
    w = S.Workload("split", B, N, Hq, Hkv, d, 64, 2, 3, dtype, 700 + d, "iid")
    t = S.make_inputs(w)
    prob = T.oracle_problem(w, t)
    dev = T.Device(w, t)
    dev.forward()
    assert dev.sync_status() == 0
    T.check_forward_dev(dev, prob, S.sample_queries(w, 200, B=B))
