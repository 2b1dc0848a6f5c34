"""Scoring in two sweeps over K (tensor cores, more than 64 rows, long units, or tasks sized by the
caller) at the sizes and head dims where its variants begin and end, against the fp64 oracle."""
import numpy as np
import pytest
import torch

from oracle import laq_oracle as orc
from test_gpu_parity import laq, rand_inputs  # noqa: F401 (laq is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [64, 80])
@pytest.mark.parametrize("W", [17, 32])         # 68 and 128 rows
def test_scores_of_other_head_dims_are_as_precise_as_fp32_sums(laq, D, W):  # noqa: F811
    # Every term is an exponential of the hardware (relative error 2^-22) of an argument rounded to fp32
    # (below 2^5, so within 2^-20 absolute, and rounding errors of different keys are independent): the
    # scores of a unit together stay within 2^-21 = 4.8e-7 of the oracle's in the 2-norm (measured: 1.0 to
    # 2.4e-7, as with fp32 arithmetic on CUDA cores).
    q, k, v = rand_inputs(1, 2, 8, 2, D, 3000, W, seed=D + W)
    out = laq.evict(q.cuda(), k.cuda(), v.cuda(), 100, want_scores=True)
    ref = orc.evict(q, k, v, W, 7, 100)["scores"]
    got = out["scores"].cpu().numpy().astype(np.float64)
    assert np.linalg.norm(got - ref) <= 4.8e-7 * np.linalg.norm(ref)
