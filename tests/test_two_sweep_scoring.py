"""Scoring in two sweeps over K (tensor cores, more than 64 rows, long units, or tasks sized by the
caller) at the sizes and head dims where its variants begin and end, against the fp64 oracle."""
import numpy as np
import pytest
import torch

from oracle import laq_oracle as orc
from parity_util import SCORE_RTOL, score_rel_err
from test_gpu_parity import compare_all_units, laq, rand_inputs  # noqa: F401 (laq is a fixture)

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


@pytest.mark.parametrize("D", [64, 80, 128])
@pytest.mark.parametrize("G,W,L", [(8, 17, 3000), (5, 32, 3000), (8, 32, 3000), (8, 32, 600)])     # 136, 160, 256 rows
@pytest.mark.parametrize("group", [0, 2])
def test_scores_of_two_row_blocks_are_as_precise_as_fp32_sums(laq, G, W, L, D, group):  # noqa: F811
    # the same bound. An eighth of sweep 1's exponentials comes from a polynomial of degree 5 on the FMA pipe:
    # the one of degree 3 that 65 to 128 rows of 128 dims take leaves 1e-6, and must not be in its place.
    # One column sum per head with a window of 17 is formed on CUDA cores.
    q, k, v = rand_inputs(1, 1, 2 * G, 2, D, L, W, seed=D + W + G)
    out = laq.evict(q.cuda(), k.cuda(), v.cuda(), 100, want_scores=True, group_mode=group)
    ref = orc.evict(q, k, v, W, 7, 100, group_mode=group)["scores"]
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


# ------------------------------------------------------------------ which kernel scores
def evict_with(laq, q, k, v, R, kernel, B, tiles_per_task=0, local_window=0, lens=None, group=0, want=None):  # noqa: F811
    """laq_evict with the scheduling knob set (a nonzero one keeps units of up to 64 rows with the two
    sweeps), in the form that compare_all_units takes. `want`: part of the name of the kernel that scores."""
    qd, kd, vd = q.cuda(), k.cuda(), v.cuda()
    NL, Bt, Hq, D = q.shape[0], q.shape[1], q.shape[2], q.shape[4]
    H = Hq if group == laq.LAQ_GROUP_PER_HEAD else k.shape[2]
    out = {"k_out": torch.empty((NL, Bt, H, B, D), dtype=torch.bfloat16, device="cuda"),
           "idx": torch.empty((NL, Bt, H, B), dtype=torch.int32, device="cuda"),
           "scores": torch.empty((NL, Bt, H, k.shape[3] - R), dtype=torch.float32, device="cuda")}
    out["v_out"] = torch.empty_like(out["k_out"])
    p = laq.params_for(qd, kd, R, kernel, B, v=vd, out=out["k_out"])
    p.tiles_per_task, p.local_window, p.group_mode = tiles_per_task, local_window, group
    p.set_seq_lens(lens)
    ws = laq.alloc_workspace(p, "cuda")

    def call():
        laq.laq_evict(p, qd, kd, vd, out["k_out"], out["v_out"], out["idx"], out["scores"], ws)
        assert laq.laq_last_device_status(p, ws) == laq.LAQ_OK
    call()
    if want is not None:
        assert want in scoring_kernels(call)
    return dict(out, params=p, ws=ws)


def scoring_kernels(call, *more):
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    names = " ".join(e.key for e in prof.key_averages())
    return {n for n in ("score_cluster_kernel", "score_tc_kernel", "simt_stats_kernel", *more) if n in names}


TWO_SWEEP = [
    # NL Bt Hq Hkv D    L     W  W_local k  B  tiles lens        group
    (1, 1, 4, 1, 8, 700, 17, 0, 3, 60, 0, None, 0),              # head dims below 128, 68 rows
    (1, 2, 8, 2, 64, 1300, 32, 16, 7, 90, 0, (1300, 401), 0),    # 128 rows
    (1, 1, 8, 1, 80, 900, 17, 17, 5, 60, 0, None, 0),            # 136 rows: two row blocks
    (1, 1, 8, 1, 112, 2300, 32, 0, 7, 100, 0, None, 0),          # 256 rows, several tasks
    (1, 1, 8, 2, 64, 1100, 32, 0, 7, 90, 0, None, 2),            # one column sum per head
    (1, 1, 4, 1, 96, 640, 64, 0, 7, 100, 0, None, 1),
    (1, 1, 2, 2, 128, 1500, 1, 0, 7, 60, 4, None, 0),            # up to 64 rows: every row held twice
    (1, 2, 8, 2, 128, 1030, 16, 8, 7, 90, 1, (1030, 129), 0),
    (2, 1, 8, 2, 64, 2500, 8, 0, 5, 90, 3, None, 0),
    (1, 1, 8, 2, 128, 1300, 16, 0, 7, 90, 4, None, 1),           # and one column sum per head
    (1, 2, 8, 2, 128, 1300, 8, 0, 7, 90, 4, (1300, 500), 2),
    (1, 1, 4, 2, 72, 900, 32, 0, 7, 90, 2, None, 2),
    (1, 1, 8, 2, 128, 16385, 16, 0, 5, 64, 0, None, 0),          # too long for a cluster's tensor memory
]


@pytest.mark.parametrize("case", TWO_SWEEP, ids=[f"D{c[4]}-M{c[2] // c[3] * c[6]}-L{c[5]}-g{c[12]}" for c in TWO_SWEEP])
def test_two_sweeps_match_oracle(laq, case):  # noqa: F811
    NL, Bt, Hq, Hkv, D, L, W, Wl, kernel, B, tiles, lens, group = case
    q, k, v = rand_inputs(NL, Bt, Hq, Hkv, D, L, W, seed=L + D + W, kscale=1.5)
    if lens is not None:
        for b, Lb in enumerate(lens):
            k[:, b, :, Lb:] = float("nan")
    out = evict_with(laq, q, k, v, W, kernel, B, tiles, Wl, lens, group, want="score_tc_kernel")
    compare_all_units(laq, q, k, v, W, kernel, B, out=out, local_window=Wl, seq_lens=lens, group_mode=group)


# More than 128 rows: a tile's two row blocks change hands on their own, so the edges are the rows of the
# second block (one group, one chunk, odd numbers of chunks), units of one to five tiles (fewer than the K
# stages, odd numbers for a pair of warpgroups), tasks of one tile, and tiles that are masked in part.
TWO_BLOCKS = [
    # NL Bt G   L     W  W_local tiles lens          group
    (1, 1, 3, 128, 43, 0, 0, None, 0),            # 129 rows, one tile
    (2, 1, 5, 257, 32, 16, 0, None, 0),           # 160 rows, two tiles and a key
    (1, 2, 7, 640, 32, 32, 1, (640, 130), 0),     # 224 rows, a task per tile, all queries local
    (1, 1, 8, 1153, 32, 0, 3, None, 0),           # 256 rows, tasks of three tiles
    (3, 2, 6, 4500, 32, 5, 0, (4500, 1000), 0),   # 192 rows, several tasks a unit
    (1, 1, 5, 900, 32, 0, 0, None, 2),            # one column sum per head, second block of one chunk
    (1, 1, 4, 1300, 64, 8, 2, None, 1),           # heads of two chunks
]


@pytest.mark.parametrize("case", TWO_BLOCKS, ids=[f"M{c[2] * c[4]}-L{c[3]}-g{c[8]}" for c in TWO_BLOCKS])
def test_two_row_blocks_match_oracle(laq, case):  # noqa: F811
    NL, Bt, G, L, W, Wl, tiles, lens, group = case
    q, k, v = rand_inputs(NL, Bt, 2 * G, 2, 128, L, W, seed=L + G, kscale=1.5)
    if lens is not None:
        for b, Lb in enumerate(lens):
            k[:, b, :, Lb:] = float("nan")
    B = W + 20
    out = evict_with(laq, q, k, v, W, 7, B, tiles, Wl, lens, group, want="score_tc_kernel")
    compare_all_units(laq, q, k, v, W, 7, B, out=out, local_window=Wl, seq_lens=lens, group_mode=group)


@pytest.mark.parametrize("W,G", [(4, 18), (4, 64), (8, 9), (8, 17), (16, 5), (16, 11), (32, 3), (32, 5), (64, 2), (64, 3)])
def test_heads_of_every_window(laq, W, G):  # noqa: F811
    # one column sum per head: every window that takes this path, with one row block (72 to 128 rows) and with
    # two, heads that end inside a chunk of 32 rows, with it, and over two, and a last chunk that is not full
    q, k, v = rand_inputs(1, 1, G, 1, 128, 700, W, seed=W + G, kscale=1.5)
    out = evict_with(laq, q, k, v, W, 7, W + 20, group=2, want="score_tc_kernel")
    compare_all_units(laq, q, k, v, W, 7, W + 20, out=out, group_mode=2)


@pytest.mark.parametrize("G,W,D", [(8, 32, 128), (5, 32, 128), (8, 17, 64), (4, 32, 128), (4, 32, 64)])
@pytest.mark.parametrize("what", [float("-inf"), float("inf"), float("nan")])
def test_row_without_a_softmax_is_not_left_out(laq, G, W, D, what):  # noqa: F811
    # every logit of one row of KV head 0 is -inf, +inf or NaN: that row's attention weights, and with them every
    # score of the head, are NaN (as in the fp64 definition), and the other head is not touched
    q, k, v = rand_inputs(1, 1, 2 * G, 2, D, 1000, W, seed=W + D)
    q[..., 0] = 0.0
    k[..., 0] = 1.0
    for row in (0, 2, G * W - 1):
        bad = q.clone()
        bad[0, 0, row // W, row % W, 0] = what
        out = evict_with(laq, bad, k, v, W, 1, W + 20)
        good = evict_with(laq, q, k, v, W, 1, W + 20)
        assert out["scores"][0, 0, 0].isnan().all()
        assert torch.equal(out["scores"][0, 0, 1], good["scores"][0, 0, 1])


# Batches of many more tasks than SMs, so that every CTA takes tasks of both sweeps and of several units in
# turn: the one Q stage, the ring of K stages and the phases of the accumulators run on across them.
MANY_TASKS = [
    # Bt G  L     W  W_local tiles ragged group
    (32, 5, 2300, 32, 0, 0, False, 0),            # 160 rows, 64 units
    (32, 8, 3000, 32, 16, 0, False, 0),           # 256 rows, local queries
    (40, 8, 1500, 32, 0, 1, True, 0),             # 256 rows, a task per tile, prompts of different lengths
    (32, 6, 4900, 32, 5, 13, True, 0),            # 192 rows, tasks of thirteen tiles, prompts of different lengths
    (32, 8, 4100, 32, 17, 5, False, 0),           # 256 rows, odd numbers of tiles a task
    (32, 8, 3500, 17, 17, 7, False, 0),           # 136 rows, likewise
    (32, 5, 2000, 32, 0, 0, True, 2),             # one column sum per head
    (32, 8, 1700, 32, 8, 3, False, 1),
]
# Many tasks of few tiles: these are handed over whole, both row blocks at once
SHORT_TASKS = [
    (100, 3, 300, 43, 0, 0, False, 0),            # 129 rows, three tiles a unit
    (100, 5, 600, 32, 16, 0, False, 0),           # 160 rows, five tiles, local queries
    (100, 8, 200, 32, 0, 0, False, 0),            # 256 rows, two tiles
    (160, 6, 2600, 32, 0, 0, False, 0),           # 192 rows, three tasks of seven tiles
    (100, 8, 900, 17, 17, 1, False, 0),           # 136 rows, a task per tile, all queries local
    (100, 5, 1500, 32, 5, 0, True, 0),            # 160 rows, prompts of different lengths
]


@pytest.mark.parametrize("case", SHORT_TASKS, ids=[f"M{c[1] * c[3]}-L{c[2]}-t{c[5]}" for c in SHORT_TASKS])
def test_two_row_blocks_handed_over_whole(laq, case):  # noqa: F811
    check_many_tasks(laq, case, whole=True)


@pytest.mark.parametrize("case", MANY_TASKS, ids=[f"M{c[1] * c[3]}-L{c[2]}-t{c[5]}-g{c[7]}" for c in MANY_TASKS])
def test_two_row_blocks_through_many_tasks(laq, case):  # noqa: F811
    check_many_tasks(laq, case, whole=case == MANY_TASKS[2])


def check_many_tasks(laq, case, whole):  # noqa: F811
    # Against the CUDA-core kernel, which a layer stride that no tensor map holds selects (with one layer it is
    # never used): fp32 sums of the same terms in other orders, 2^-21 in the 2-norm apiece.
    Bt, G, L, W, Wl, tiles, ragged, group = case
    Hkv, D = 2, 128
    g = torch.Generator(device="cuda").manual_seed(L)
    q = torch.randn((1, Bt, G * Hkv, W, D), generator=g, device="cuda", dtype=torch.bfloat16)
    k = torch.randn((1, Bt, Hkv, L, D), generator=g, device="cuda", dtype=torch.bfloat16)
    lens = [L - b * (L - 2 * W) // Bt for b in range(Bt)] if ragged else None
    for b, Lb in enumerate(lens or ()):
        k[:, b, :, Lb:] = float("nan")
    p = laq.params_for(q, k, W, 1, W + 20)
    p.tiles_per_task, p.local_window, p.group_mode = tiles, Wl, group
    p.set_seq_lens(lens)
    got = torch.zeros((1, Bt, Hkv * (G if group == 2 else 1), L - W), device="cuda")
    want = torch.zeros_like(got)
    ws = laq.alloc_workspace(p, "cuda")

    def call():
        laq.laq_score(p, q, k, got, ws)
    assert scoring_kernels(call, "score_tc_kernel<false, true, false, 0, false>") == (
        {"score_tc_kernel", "score_tc_kernel<false, true, false, 0, false>"} if whole else {"score_tc_kernel"})
    for _ in range(3):
        call()
        assert laq.laq_last_device_status(p, ws) == laq.LAQ_OK
        p.k_stride_layer, stride = 1 << 40, p.k_stride_layer
        laq.laq_score(p, q, k, want, ws)
        p.k_stride_layer = stride
        assert not got.isnan().any() and float((got - want).norm() / want.norm()) < 1e-6


CUDA_CORES = [
    (1, 1, 3, 1, 136, 500, 32, 0, 7, 60, None, 0),               # head dims above 128 with more than 64 rows
    (1, 2, 8, 2, 192, 900, 32, 16, 5, 90, (900, 333), 0),
    (1, 1, 8, 1, 256, 300, 32, 32, 7, 64, None, 0),              # 256 rows of 256 dims
    (1, 1, 8, 1, 128, 700, 9, 0, 7, 60, None, 1),                # windows that straddle the groups of four rows
    (1, 2, 4, 1, 128, 1200, 25, 5, 3, 60, (1200, 130), 2),
    (1, 1, 8, 2, 200, 600, 20, 0, 7, 60, None, 2),
]


@pytest.mark.parametrize("case", CUDA_CORES, ids=[f"D{c[4]}-M{c[2] // c[3] * c[6]}-g{c[11]}" for c in CUDA_CORES])
def test_cuda_cores_match_oracle(laq, case):  # noqa: F811
    NL, Bt, Hq, Hkv, D, L, W, Wl, kernel, B, lens, group = case
    q, k, v = rand_inputs(NL, Bt, Hq, Hkv, D, L, W, seed=L + D + W, kscale=1.5)
    if lens is not None:
        for b, Lb in enumerate(lens):
            k[:, b, :, Lb:] = float("nan")
    out = evict_with(laq, q, k, v, W, kernel, B, 0, Wl, lens, group, want="simt_stats_kernel")
    compare_all_units(laq, q, k, v, W, kernel, B, out=out, local_window=Wl, seq_lens=lens, group_mode=group)
    # and on the library's own scratch, whose last contents another problem left there
    if group == 0:
        qd, kd = q.cuda(), k.cuda()
        got = torch.full_like(out["scores"], float("nan"))
        laq.laq_score_static(out["params"], qd, kd, got)
        assert torch.equal(got, out["scores"])


def test_layout_that_tma_cannot_describe_is_scored_on_cuda_cores(laq):  # noqa: F811
    # strides of 2^40 bytes and more are beyond a tensor map; with one layer the stride is never used
    for W in (8, 32):
        q, k, v = rand_inputs(1, 1, 8, 2, 128, 500, W, seed=W, kscale=1.5)
        out = laq.evict(q.cuda(), k.cuda(), v.cuda(), 70, want_scores=True)
        p, qd, kd = out["params"], q.cuda(), k.cuda()
        p.k_stride_layer = 1 << 40
        got = torch.zeros_like(out["scores"])

        def call():
            laq.laq_score(p, qd, kd, got, out["ws"])
        call()
        assert "simt_stats_kernel" in scoring_kernels(call)
        want = orc.evict(q, k, None, W, 7, 70, want_idx=False)["scores"]
        assert score_rel_err(got.cpu().numpy(), want) <= SCORE_RTOL


@pytest.mark.parametrize("W,G,tiles", [(16, 4, 4), (2, 4, 8), (32, 4, 0), (32, 8, 0)])
def test_extreme_logits_and_late_maximum_in_two_sweeps(laq, W, G, tiles):  # noqa: F811
    # logits of +-hundreds and a very large key late in the prompt: the reference of sweep 1 has to move
    # several times, also in the middle of a task, and sweep 2 sees probabilities below the smallest normal
    Hkv, D, L, kernel, B = 2, 128, 4200, 7, 150
    g = torch.Generator().manual_seed(404 + W)
    q = torch.randn((1, 1, G * Hkv, W, D), generator=g).to(torch.bfloat16)
    k = (torch.randn((1, 1, Hkv, L, D), generator=g) * 12.0).to(torch.bfloat16)
    v = torch.randn((1, 1, Hkv, L, D), generator=g).to(torch.bfloat16)
    for h in range(Hkv):
        qbar = q[0, 0, h * G:(h + 1) * G].float().mean(dim=(0, 1))
        k[0, 0, h, 3900] = (qbar * 60.0).to(torch.bfloat16)
    for Wl in (0, min(W, 1)):
        out = evict_with(laq, q, k, v, W, kernel, B, tiles, Wl, want="score_tc_kernel")
        compare_all_units(laq, q, k, v, W, kernel, B, out=out, local_window=Wl)
