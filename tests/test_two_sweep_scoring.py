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


@pytest.mark.parametrize("W", [8, 32])          # 32 and 128 rows
def test_one_workspace_serves_batches_of_other_lengths(laq, W):  # noqa: F811
    # sized for the allocated batch, then used for batches of shorter prompts and for fewer layers: the
    # sizes lie on either side of where tasks of 8 and of 16 tiles are chosen (12032 .. 48128 tiles)
    NL, Bt, Hkv, D, L, B = 16, 4, 8, 128, 12001, 200
    g = torch.Generator(device="cuda").manual_seed(W)
    q = torch.randn((NL, Bt, 4 * Hkv, W, D), generator=g, device="cuda", dtype=torch.bfloat16)
    k = torch.randn((NL, Bt, Hkv, L, D), generator=g, device="cuda", dtype=torch.bfloat16)
    ws = laq.alloc_workspace(laq.params_for(q, k, W, 7, B), "cuda")
    for n, lens in ((NL, None), (NL, (12001, 8771, 5541, 2311)), (NL, (12001,) * 4), (NL, (201,) * 4), (12, None),
                    (12, (12001,) * 4), (4, None)):
        p = laq.params_for(q[:n], k[:n], W, 7, B)
        p.set_seq_lens(lens)
        scores = torch.empty((n, Bt, Hkv, L - W), dtype=torch.float32, device="cuda")
        assert laq.laq_score(p, q[:n], k[:n], scores, ws, check=False) == laq.LAQ_OK
        assert laq.laq_last_device_status(p, ws) == laq.LAQ_OK
        own = torch.empty_like(scores)
        laq.laq_score(p, q[:n], k[:n], own, laq.alloc_workspace(p, "cuda"))
        # (which softmax warps take a tile depends on the tiles their CTA has had before, so the order of a
        # sum is not fixed where tasks have odd numbers of tiles: fp32 rounding only)
        assert float((scores - own).norm() / own.norm()) < 5e-7


def test_static_scratch_takes_longer_tasks_where_shorter_ones_do_not_fit(laq):  # noqa: F811
    # 256 rows and 16384 keys: 97 KB of scratch a unit with tasks of 8 tiles, 81 KB with tasks of 16, so that
    # 92 units fit the fixed 8 MB only with the latter, which the caller's workspace would not need
    NL, Hkv, D, L, W, B = 23, 4, 128, 16384, 32, 100
    g = torch.Generator(device="cuda").manual_seed(5)
    q = torch.randn((NL, 1, 8 * Hkv, W, D), generator=g, device="cuda", dtype=torch.bfloat16)
    k = torch.randn((NL, 1, Hkv, L, D), generator=g, device="cuda", dtype=torch.bfloat16)
    p = laq.params_for(q, k, W, 7, B)
    want = torch.empty((NL, 1, Hkv, L - W), dtype=torch.float32, device="cuda")
    laq.laq_score(p, q, k, want, laq.alloc_workspace(p, "cuda"))
    got = torch.full_like(want, float("nan"))
    assert laq.laq_score_static(p, q, k, got, check=False) == laq.LAQ_OK
    # the same terms, the row sums added in other groups: fp32 rounding only
    assert float((got - want).norm() / want.norm()) < 5e-7
    # and what does not fit even so (108 units) is refused
    p = laq.make_params(27, 1, 8 * Hkv, Hkv, D, L, W, W, 7, B)
    assert laq.laq_score_static(p, q, k, got, check=False) == laq.LAQ_ERR_WORKSPACE
