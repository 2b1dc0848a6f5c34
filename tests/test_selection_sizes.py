"""Selection at the sizes where its kernels change or end: few short units (8 scores per thread), many
units (32 per thread), units of two thread blocks, and the longest that registers hold; against the
oracle's selection on the same scores, bit for bit."""
import numpy as np
import pytest
import torch

from oracle import laq_oracle as orc
from test_gpu_parity import compare_all_units, laq, rand_inputs  # noqa: F401 (laq is a fixture)

pytestmark = pytest.mark.gpu


def scores_of(kind, U, Ls, rng):
    if kind == "random":
        return rng.random((U, Ls)).astype(np.float32)
    if kind == "ties":
        return (rng.integers(0, 5, (U, Ls)) * 0.25).astype(np.float32)
    if kind == "signed":
        return rng.standard_normal((U, Ls)).astype(np.float32)
    return np.full((U, Ls), 0.125, np.float32)


@pytest.mark.parametrize("U,Ls", [(1, 2), (3, 33), (2, 1023), (148, 257), (149, 257), (2, 8192), (2, 8193),
                                  (160, 4097), (1, 32768), (1, 32769), (2, 65536), (1, 65537)])
def test_select_at_the_edges_of_its_kernels(laq, U, Ls):
    rng = np.random.default_rng(Ls + U)
    for kind in ("random", "ties", "const", "signed"):
        s = scores_of(kind, U, Ls, rng)
        for Kb in sorted({1, max(1, Ls // 3), Ls - 1}):
            R = 3
            L, B = Ls + R, Kb + R
            p = laq.make_params(1, U, 1, 1, 128, L, 1, R, 1, B)
            idx = torch.full((U, B), -1, dtype=torch.int32, device="cuda")
            laq.laq_select(p, torch.from_numpy(s).cuda(), idx)
            got = idx.cpu().numpy()
            for u in {0, U // 2, U - 1}:
                want = orc.select(s[u], L, R, B, sorted_variant=True)
                assert (got[u] == want).all(), (kind, Kb, u)


@pytest.mark.parametrize("kernel", [1, 3, 9, 65, 67])
@pytest.mark.parametrize("mode", [0, 1])
def test_pooling_inside_the_selection_equals_pooling_alone(laq, kernel, mode):
    # several scores per thread on either side of every edge; windows wider than what is staged
    for NL, L, B in ((1, 1001, 60), (40, 997, 60), (1, 33000, 700)):
        q, k, v = rand_inputs(NL, 1, 8, 4, 128, L, 2, seed=kernel + L, kscale=1.5)
        if NL == 1 and L < 2000:
            compare_all_units(laq, q, k, v, 2, kernel, B, pool_mode=mode)
        q, k, v = q.cuda(), k.cuda(), v.cuda()
        out = laq.evict(q, k, v, B, pool_kernel=kernel, keep_tail=2, want_scores=True, pool_mode=mode)
        alone = torch.empty_like(out["scores"])
        laq.laq_score(out["params"], q, k, alone, out["ws"])
        idx = torch.empty_like(out["idx"])
        laq.laq_select(out["params"], alone, idx)
        assert torch.equal(alone, out["scores"]) and torch.equal(idx, out["idx"])


@pytest.mark.parametrize("kernel", [11, 63, 101, 1999])
@pytest.mark.parametrize("mode", [0, 1])
def test_wide_pooling_windows(laq, kernel, mode):
    # one load per tap: windows inside what is staged around a CTA's positions, beyond it, and wider than
    # the short units themselves; ragged too, where a unit ends inside the row
    test_pooling_inside_the_selection_equals_pooling_alone(laq, kernel, mode)
    q, k, v = rand_inputs(1, 3, 8, 2, 128, 1500, 8, seed=kernel, kscale=1.5)
    compare_all_units(laq, q, k, v, 8, kernel, 50, pool_mode=mode, seq_lens=(1500, 1497, 61))
