"""Recall of one selection against another at the sizes where its kernels change: a warp or a block per
unit, the known set staged in shared memory or not; against numpy's intersection, exactly."""
import numpy as np
import pytest
import torch

from test_gpu_parity import laq  # noqa: F401 (a fixture)

pytestmark = pytest.mark.gpu


def ascending(rng, U, n, top):
    return np.stack([np.sort(rng.choice(top, n, replace=False)) for _ in range(U)]).astype(np.int32)


@pytest.mark.parametrize("U,n_pred,n_gold", [
    (1, 1, 1), (3, 33, 17), (2, 300, 12280), (2, 300, 12281), (2, 300, 12288), (2, 300, 12289), (1, 5, 12280),
    (1184, 64, 64), (1185, 64, 64), (5000, 7, 31), (1300, 512, 512), (1300, 513, 40), (1300, 16, 12288),
    (2700, 7, 31), (2900, 7, 31), (12001, 257, 40), (12001, 259, 40), (3900, 7, 31), (4003, 7, 31), (5757, 64, 64), (9001, 249, 40), (9001, 251, 40), (1301, 16, 12280), (300, 16, 12280)])
def test_recall_at_the_edges_of_its_kernels(laq, U, n_pred, n_gold):  # noqa: F811
    rng = np.random.default_rng(U + n_gold)
    top = 2 * max(n_pred, n_gold)
    distinct = min(U, 50)
    pred, gold = ascending(rng, distinct, n_pred, top), ascending(rng, distinct, n_gold, top)
    turn = np.arange(U) % distinct
    rec, common = laq.laq_recall(torch.from_numpy(pred[turn]).cuda(), torch.from_numpy(gold[turn]).cuda())
    want = np.array([len(np.intersect1d(a, g)) for a, g in zip(pred, gold)], np.int32)[turn]
    assert (common.cpu().numpy() == want).all()
    assert (rec.cpu().numpy() == want.astype(np.float32) / np.float32(n_gold)).all()
