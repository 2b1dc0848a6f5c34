"""Scoring with the logits of a unit kept in the tensor memory of a thread-block cluster (up to 64
softmax rows): the sizes at which tiles, row groups, clusters and head dims end, against the fp64
oracle with the tolerances of the other parity tests."""
import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from parity_util import SCORE_RTOL
from test_gpu_parity import compare_all_units, laq, rand_inputs, run_evict  # noqa: F401 (laq is a fixture)
from test_timeout_path import hooked_library

pytestmark = pytest.mark.gpu

CASES = [
    # NL Bt Hq Hkv D    L     W  W_local k  B   lens
    (1, 1, 1, 1, 128, 129, 1, 0, 1, 10, None),           # one row; a tile and one key
    (1, 1, 1, 1, 128, 128, 9, 3, 3, 20, None),           # nine rows (two groups), exactly one tile
    (1, 2, 5, 1, 128, 2049, 8, 8, 7, 100, None),         # 40 rows; 17 tiles, every CTA but one short
    (1, 1, 7, 1, 128, 1000, 8, 0, 5, 60, None),          # 56 rows run as 64
    (1, 1, 3, 1, 128, 3000, 19, 19, 7, 100, None),       # 57 rows, heads straddle the groups, all local
    (1, 1, 8, 2, 128, 16384, 16, 0, 5, 64, None),        # the longest unit that fits at 64 rows
    (1, 1, 8, 2, 128, 16385, 16, 16, 5, 64, None),       # and the first that does not
    (1, 3, 8, 2, 128, 4100, 16, 16, 7, 50, (4100, 51, 130)),  # CTAs without a tile of the short prompts
    (3, 7, 8, 2, 128, 700, 4, 2, 3, 40, None),           # more units than clusters: several rounds
    (1, 1, 4, 1, 8, 300, 4, 0, 3, 40, None),             # head dims 8 .. 256
    (1, 1, 4, 1, 80, 900, 8, 4, 7, 60, None),
    (1, 2, 4, 1, 96, 500, 16, 0, 7, 60, (500, 257)),
    (1, 1, 8, 2, 192, 1100, 8, 0, 7, 60, None),
    (1, 1, 8, 2, 256, 2000, 16, 16, 7, 60, None),
]


@pytest.mark.parametrize("case", CASES, ids=[f"L{c[5]}-M{c[2] // c[3] * c[6]}-D{c[4]}" for c in CASES])
def test_cluster_scoring_edges(laq, case):
    NL, Bt, Hq, Hkv, D, L, W, Wl, kernel, B, lens = case
    q, k, v = rand_inputs(NL, Bt, Hq, Hkv, D, L, W, seed=L + D + W, kscale=1.5)
    if lens is not None:
        for b, Lb in enumerate(lens):
            k[:, b, :, Lb:] = float("nan")
    compare_all_units(laq, q, k, v, W, kernel, B, local_window=Wl, seq_lens=lens)


@pytest.mark.parametrize("W", [1, 3, 6, 16])
def test_cluster_scoring_per_head(laq, W):
    # heads of any length; W = 16 ends inside a group of eight rows only at its end
    q, k, v = rand_inputs(1, 1, 8, 2, 128, 1300, W, seed=W, kscale=1.5)
    for mode in (1, 2):
        compare_all_units(laq, q, k, v, W, 7, 80, group_mode=mode)


def test_cluster_scoring_sums_that_overflow(laq):
    # Every warp takes the logits of its first key as reference. Here those lie 120 nats below the
    # largest key, so the sums of a warp overflow and are taken again from the true maximum.
    NL, Bt, Hq, Hkv, D, L, W, kernel, B = 1, 1, 4, 1, 128, 1100, 4, 7, 90
    q, k, v = rand_inputs(NL, Bt, Hq, Hkv, D, L, W, seed=17)
    q[..., 0] = 12.0
    k[..., 0] = 0.0
    k[:, :, :, ::32, 0] = -56.0                    # logit -59
    for j in (5, 300, 700):
        k[:, :, :, j, 0] = 56.0                    # logit +59
    err, _ = compare_all_units(laq, q, k, v, W, kernel, B)
    assert err < SCORE_RTOL
    out = laq.evict(q.cuda(), k.cuda(), v.cuda(), B, pool_kernel=kernel)
    assert {5, 300, 700} <= set(out["idx"][0, 0, 0].tolist())
    assert np.isfinite(out["k_out"].float().cpu().numpy()).all()


def launched_cluster(laq, q, k, R, kernel, B, group=0):  # noqa: F811
    """CTAs per cluster of a scoring call of these sizes (0: another kernel takes it)."""
    p = laq.params_for(q, k, R, kernel, B)
    p.group_mode = group
    ws = laq.alloc_workspace(p, "cuda")
    H = q.shape[2] if group == 2 else k.shape[2]
    scores = torch.empty((q.shape[0], q.shape[1], H, k.shape[3] - R), device="cuda")
    hooked = hooked_library()
    assert hooked.laq_score(ctypes.byref(p), q.cuda().data_ptr(), k.cuda().data_ptr(), scores.data_ptr(), ws.data_ptr(),
                            ws.numel(), torch.cuda.current_stream().cuda_stream) == laq.LAQ_OK
    torch.cuda.synchronize()
    return hooked.laq_test_last_cluster()


# clusters whose CTAs hold several tiles of a unit (layers, batch, keys, size): six with three tiles, sixteen with four
SIZES = [(4, 2, 2000, 6), (1, 1, 8192, 16)]


@pytest.mark.parametrize("NL,Bt,L,C", SIZES)
@pytest.mark.parametrize("G,W,group", [(4, 4, 0), (4, 16, 0), (3, 19, 0), (8, 8, 2), (4, 3, 2)])
def test_sums_that_overflow_in_clusters_of(laq, NL, Bt, L, C, G, W, group):
    # as above, every warp with more than one tile: its reference lies 120 nats below the largest key, in
    # some warps in their first tile and in some in a later one
    Hkv, D, kernel, B = 2, 128, 7, W + 90
    q, k, v = rand_inputs(NL, Bt, G * Hkv, Hkv, D, L, W, seed=L + W)
    q[..., 0] = 12.0
    k[..., 0] = 0.0
    k[:, :, :, ::32, 0] = -56.0
    for j in (5, 300, 1500, L - 200):
        k[:, :, :, j, 0] = 56.0
    assert launched_cluster(laq, q, k, W, kernel, B, group) == C
    err, _ = compare_all_units(laq, q, k, v, W, kernel, B, group_mode=group)
    assert err < SCORE_RTOL


@pytest.mark.parametrize("NL,Bt,L,C", SIZES)
@pytest.mark.parametrize("W,G", [(1, 4), (3, 4), (5, 8), (6, 4), (8, 7), (16, 4)])
def test_cluster_scoring_per_head_with_several_tiles(laq, NL, Bt, L, C, W, G):
    q, k, v = rand_inputs(NL, Bt, 2 * G, 2, 128, L, W, seed=L + W, kscale=1.5)
    for mode in (1, 2):
        assert launched_cluster(laq, q, k, W, 7, 80, mode) == C
        compare_all_units(laq, q, k, v, W, 7, 80, group_mode=mode)


@pytest.mark.parametrize("G,W,group", [(1, 5, 0), (4, 2, 0), (4, 16, 0), (7, 8, 0), (4, 8, 1), (4, 3, 2)])
@pytest.mark.parametrize("what", [float("inf"), float("nan")])
def test_row_without_a_softmax_is_not_left_out_of_a_cluster(laq, G, W, group, what):
    # every logit of one row of KV head 0 is +inf or NaN: its attention weights, and with them every score
    # that adds or compares them, are NaN (as in the fp64 definition); the other KV head is not touched. Pass 2
    # takes rows 2 and 3 of every four on another pipe than rows 0 and 1.
    q, k, v = rand_inputs(1, 1, 2 * G, 2, 128, 1000, W, seed=W + G)
    q[..., 0] = 0.0
    k[..., 0] = 1.0
    H = G if group == 2 else 1
    good = run_evict(laq, q, k, v, W, 1, W + 20, group_mode=group)["scores"]
    for row in sorted({0, 1, 2, 3, G * W - 2, G * W - 1} & set(range(G * W))):
        bad = q.clone()
        bad[0, 0, row // W, row % W, 0] = what
        got = run_evict(laq, bad, k, v, W, 1, W + 20, group_mode=group)["scores"]
        nan = got[0, 0].isnan()
        if group == 1:                       # (the larger of a NaN and a number is the number)
            assert torch.equal(got[0, 0, 1], good[0, 0, 1])
        elif group == 2:
            assert nan[row // W].all()
            others = [h for h in range(2 * G) if h != row // W]
            assert torch.equal(got[0, 0, others], good[0, 0, others])
        else:
            assert nan[0].all() and torch.equal(got[0, 0, H:], good[0, 0, H:])


@pytest.mark.parametrize("W,L,lens", [(1, 128, None), (2, 700, None), (4, 500, tuple([500, 131] * 16))])
def test_cluster_scoring_many_short_units_of_few_rows(laq, W, L, lens):
    # At most 32 rows: one of the two exchange warps has no row of its own. Three and more units fit the
    # tensor memory at once, so the other one can be that far ahead; the two must stay in step.
    NL, Bt, Hq, Hkv, D, kernel, B = 4, 32, 16, 4, 128, 3, 24
    q, k, v = rand_inputs(NL, Bt, Hq, Hkv, D, L, W, seed=W + L, kscale=1.5)
    compare_all_units(laq, q, k, v, W, kernel, B, seq_lens=lens)
    qc, kc, vc = q.cuda(), k.cuda(), v.cuda()
    first = laq.evict(qc, kc, vc, B, pool_kernel=kernel, want_scores=True, seq_lens=lens)
    for _ in range(50):
        out = laq.evict(qc, kc, vc, B, pool_kernel=kernel, want_scores=True, seq_lens=lens, ws=first["ws"])
    assert laq.laq_last_device_status(out["params"], out["ws"]) == laq.LAQ_OK
    assert torch.equal(out["scores"], first["scores"]) and torch.equal(out["idx"], first["idx"])


@pytest.mark.parametrize("units,G,W,D,L,lens,group,C", [
    # between the powers of two
    (256, 4, 16, 128, 2500, None, 0, 5),                 # four tiles a CTA
    (256, 4, 16, 128, 6007, None, 0, 6),                 # all slots of the tensor memory
    (256, 4, 16, 128, 9000, None, 0, 9),
    (64, 4, 12, 128, 3000, None, 0, 6),
    (16, 2, 4, 64, 6646, None, 0, 6),
    (40, 5, 8, 128, 3000, None, 2, 6),                   # one sum per head
    # powers of two
    (256, 4, 16, 128, 9000, (9000, 5001, 1153, 129), 0, 16),   # (prompts of different lengths take no other)
    (256, 4, 16, 128, 4096, None, 0, 8),
    (1184, 4, 16, 128, 384, None, 0, 1),                 # many rounds of short units: bound by the chain from a unit's
    (512, 4, 4, 128, 582, None, 0, 1),                   # first MMA to the end of its pass 2, which a cluster does
    (256, 1, 4, 96, 539, None, 0, 1),                    # not shorten
    (224, 8, 8, 128, 639, None, 2, 1),
    (896, 4, 12, 128, 555, None, 0, 2),
    (56, 4, 8, 128, 2218, None, 0, 4),
])
def test_clusters_of_any_size(laq, units, G, W, D, L, lens, group, C):
    # against the other tensor-core kernel (which a task size set by the caller selects). Both sum the same
    # exponentials, arguments rounded to fp32, in other orders: 2^-21 in the 2-norm apiece.
    Bt, Hkv = (len(lens) if lens else 1), 8
    NL = units // (Bt * Hkv)
    g = torch.Generator(device="cuda").manual_seed(L)
    q = torch.randn((NL, Bt, G * Hkv, W, D), generator=g, device="cuda", dtype=torch.bfloat16)
    k = torch.randn((NL, Bt, Hkv, L, D), generator=g, device="cuda", dtype=torch.bfloat16)
    p = laq.params_for(q, k, W, 1, W + 20)
    p.set_seq_lens(lens)
    p.group_mode = group
    got = torch.full((NL, Bt, Hkv * (G if group == 2 else 1), L - W), float("nan"), device="cuda")
    ws = laq.alloc_workspace(p, "cuda")
    laq.laq_score(p, q, k, got, ws)
    assert laq.laq_last_device_status(p, ws) == laq.LAQ_OK
    hooked = hooked_library()               # (the same code, and says which size it launched)
    again = torch.full_like(got, float("nan"))
    assert hooked.laq_score(ctypes.byref(p), q.data_ptr(), k.data_ptr(), again.data_ptr(), ws.data_ptr(), ws.numel(),
                            torch.cuda.current_stream().cuda_stream) == laq.LAQ_OK
    assert hooked.laq_test_last_cluster() == C
    assert torch.equal(got, again)
    p.tiles_per_task = 8
    want = torch.empty_like(got)
    laq.laq_score(p, q, k, want, laq.alloc_workspace(p, "cuda"))
    assert float((got - want).norm() / want.norm()) < 1e-6


FIRST_USE = """
import sys
sys.path.insert(0, {root!r})
import torch
from paper_2505_20334_b200 import binding as laq
g = torch.Generator(device="cuda").manual_seed(1)
def problem(L, group):
    q = torch.randn((4, 1, 8, 8, 128), generator=g, device="cuda", dtype=torch.bfloat16)
    k = torch.randn((4, 1, 2, L, 128), generator=g, device="cuda", dtype=torch.bfloat16)
    p = laq.params_for(q, k, 8, 7, 40)
    p.group_mode = group
    s = torch.full((4, 1, 8 if group == 2 else 2, L - 8), float("nan"), device="cuda")
    return p, q, k, s, laq.alloc_workspace(p, "cuda")
laq.laq_score(*problem(512, 0))                 # a cluster of 4 CTAs: the library is up
for group in (0, 2):
    p, q, k, s, ws = problem(1100, group)       # of 9
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        laq.laq_score(p, q, k, s, ws)
    assert s.isnan().all()                      # captured, not run
    graph.replay()
    torch.cuda.synchronize()
    assert laq.laq_last_device_status(p, ws) == laq.LAQ_OK
    again = torch.empty_like(s)
    laq.laq_score(p, q, k, again, ws)
    assert torch.equal(s, again)
"""


def test_first_use_of_a_cluster_size_may_be_captured():
    # the kernels of sizes between the powers of two are loaded when first wanted, also under a capture
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", FIRST_USE.format(root=root)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
