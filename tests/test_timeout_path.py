"""The bounded device-side waits of the scoring kernels, exercised the only way that is safe on a
shared GPU: a wait is made to run out by a flag that nothing sets. A copy of the library built with
a test hook and a ~1.5 ms wait limit withholds the row statistics of one unit; whoever waits for
them (the unit's second sweep, or the other CTAs of its cluster) gives up, the whole kernel returns, the host reads
LAQ_ERR_TIMEOUT, and the next ordinary call on the same workspace works. Nothing traps or faults."""
import ctypes

import numpy as np
import pytest
import torch

from parity_util import SCORE_RTOL, score_rel_err

pytestmark = pytest.mark.gpu


def hooked_library():
    """A copy of the library with the test hooks and a ~1.5 ms limit on every wait."""
    from paper_2505_20334_b200 import binding as laq
    from paper_2505_20334_b200 import build

    build.build_liblaq()
    hooked = laq.load_library(build.build_liblaq(
        defines=["-DLAQ_TEST_HOOKS", "-DLAQ_TIMEOUT_CYCLES=3000000LL"], variant="hooks"))
    for f in (hooked.laq_test_withhold_unit, hooked.laq_test_withhold_launches):
        f.argtypes, f.restype = [ctypes.c_longlong], None
    return hooked


def test_wait_that_runs_out_is_reported_and_the_context_stays_usable():
    from paper_2505_20334_b200 import binding as laq
    from paper_2505_20334_b200 import build
    from oracle import laq_oracle as orc

    build.build_liblaq()
    hooked = laq.load_library(build.build_liblaq(
        defines=["-DLAQ_TEST_HOOKS", "-DLAQ_TIMEOUT_CYCLES=3000000LL"], variant="hooks"))
    hooked.laq_test_withhold_unit.argtypes = [ctypes.c_longlong]
    hooked.laq_test_withhold_unit.restype = None

    NL, Bt, Hq, Hkv, D, L, W, R, kernel, B = 1, 1, 8, 2, 128, 1024, 16, 16, 7, 100
    g = torch.Generator().manual_seed(9)
    q = torch.randn((NL, Bt, Hq, W, D), generator=g).to(torch.bfloat16).cuda()
    k = torch.randn((NL, Bt, Hkv, L, D), generator=g).to(torch.bfloat16).cuda()
    p = laq.params_for(q, k, R, kernel, B)
    ws = laq.alloc_workspace(p, "cuda")
    scores = torch.zeros((NL, Bt, Hkv, L - R), dtype=torch.float32, device="cuda")
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)

    def score(lib):
        return lib.laq_score(ctypes.byref(p), ctypes.c_void_p(q.data_ptr()), ctypes.c_void_p(k.data_ptr()),
                             ctypes.c_void_p(scores.data_ptr()), ctypes.c_void_p(ws.data_ptr()),
                             ws.numel(), stream)

    def status(lib):
        return lib.laq_last_device_status(ctypes.byref(p), ctypes.c_void_p(ws.data_ptr()), ws.numel(), stream)

    # unit 1 never publishes its statistics: the wait for them runs out
    hooked.laq_test_withhold_unit(1)
    try:
        assert score(hooked) == laq.LAQ_OK          # the call itself only enqueues
        assert status(hooked) == laq.LAQ_ERR_TIMEOUT
    finally:
        hooked.laq_test_withhold_unit(-1)
    assert torch.cuda.is_available() and torch.zeros(1, device="cuda").item() == 0  # context alive
    # the same build, hook off, same workspace: an ordinary run
    assert score(hooked) == laq.LAQ_OK
    assert status(hooked) == laq.LAQ_OK
    again = scores.clone()
    # and the shipped library gives the same bits
    scores.zero_()
    assert score(laq.lib) == laq.LAQ_OK and status(laq.lib) == laq.LAQ_OK
    assert torch.equal(again, scores)
    ref = orc.evict(q.cpu(), k.cpu(), None, R, kernel, B, want_idx=False)["scores"]
    assert score_rel_err(scores.cpu().numpy(), ref) <= SCORE_RTOL


@pytest.mark.parametrize("W", [16, 32])     # 64 rows: one sweep in a cluster; 128 rows: two sweeps
def test_wait_that_runs_out_in_one_piece_of_a_host_call_is_reported(W):
    # a host cache large enough to be taken in two pieces of layers; only the first one's scoring gives up
    from paper_2505_20334_b200 import binding as laq

    hooked = hooked_library()
    NL, Bt, Hq, Hkv, D, L, kernel, B = 2, 1, 8, 2, 128, 8192, 7, 100     # 8.4 MB of keys
    g = torch.Generator().manual_seed(W)
    q = torch.randn((NL, Bt, Hq, W, D), generator=g).to(torch.bfloat16).pin_memory()
    k, v = (torch.randn((NL, Bt, Hkv, L, D), generator=g).to(torch.bfloat16).pin_memory() for _ in range(2))
    he = laq.HostEvictor(tuple(q.shape), tuple(k.shape), B, kernel, W, "cuda")
    p = ctypes.byref(he.params)
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)

    def run():
        assert hooked.laq_evict_host(p, q.data_ptr(), k.data_ptr(), v.data_ptr(), he.h_k_out.data_ptr(),
                                     he.h_v_out.data_ptr(), he.h_idx.data_ptr(), he.staging.data_ptr(),
                                     he.staging.numel(), he.ws.data_ptr(), he.ws.numel(), stream) == laq.LAQ_OK
        return hooked.laq_last_device_status(p, he.ws.data_ptr(), he.ws.numel(), stream)

    assert run() == laq.LAQ_OK and hooked.laq_last_launch_count() > 3      # two pieces
    want = he.h_idx.clone()
    hooked.laq_test_withhold_unit(1)
    hooked.laq_test_withhold_launches(1)
    try:
        assert run() == laq.LAQ_ERR_TIMEOUT
    finally:
        hooked.laq_test_withhold_unit(-1)
        hooked.laq_test_withhold_launches(-1)
    assert run() == laq.LAQ_OK and torch.equal(he.h_idx, want)             # the next call starts afresh


@pytest.mark.parametrize("G,W,tiles,group", [(4, 16, 2, 0), (4, 32, 0, 0), (8, 32, 0, 0), (4, 32, 0, 2), (4, 16, 0, 2)])
def test_wait_that_runs_out_in_the_other_scoring_kernels(G, W, tiles, group):
    # two sweeps with every row held twice (64 rows, tasks sized by the caller), 128 and 256 rows, one column
    # sum per head; and the cluster kernel with one column sum per head
    from paper_2505_20334_b200 import binding as laq

    hooked = hooked_library()
    NL, Bt, Hkv, D, L, kernel, B = 1, 1, 2, 128, 1024, 7, 100
    g = torch.Generator().manual_seed(W)
    q = torch.randn((NL, Bt, G * Hkv, W, D), generator=g).to(torch.bfloat16).cuda()
    k = torch.randn((NL, Bt, Hkv, L, D), generator=g).to(torch.bfloat16).cuda()
    p = laq.params_for(q, k, W, kernel, B)
    p.tiles_per_task, p.group_mode = tiles, group
    ws = laq.alloc_workspace(p, "cuda")
    scores = torch.zeros((NL, Bt, Hkv * (G if group == 2 else 1), L - W), dtype=torch.float32, device="cuda")
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)

    def run(lib):
        assert lib.laq_score(ctypes.byref(p), q.data_ptr(), k.data_ptr(), scores.data_ptr(), ws.data_ptr(),
                             ws.numel(), stream) == laq.LAQ_OK
        return lib.laq_last_device_status(ctypes.byref(p), ws.data_ptr(), ws.numel(), stream)

    assert run(hooked) == laq.LAQ_OK
    want = scores.clone()
    hooked.laq_test_withhold_unit(1)
    try:
        assert run(hooked) == laq.LAQ_ERR_TIMEOUT
    finally:
        hooked.laq_test_withhold_unit(-1)
    for lib in (hooked, laq.lib):
        scores.zero_()
        assert run(lib) == laq.LAQ_OK
        assert torch.equal(scores, want)


@pytest.mark.parametrize("G,W", [(1, 8), (2, 8), (3, 8), (4, 8), (5, 8), (6, 8), (8, 8)])   # every group of eight rows
@pytest.mark.parametrize("NL,Bt,L,C", [(4, 2, 2000, 6), (1, 1, 8192, 16)])
@pytest.mark.parametrize("group", [0, 2])
def test_wait_that_runs_out_in_clusters(G, W, NL, Bt, L, C, group):
    # every variant of the cluster kernel, for a size between the powers of two and for one of them
    from paper_2505_20334_b200 import binding as laq

    hooked = hooked_library()
    Hkv, D = 2, 128
    g = torch.Generator(device="cuda").manual_seed(G + L)
    q = torch.randn((NL, Bt, G * Hkv, W, D), generator=g, device="cuda", dtype=torch.bfloat16)
    k = torch.randn((NL, Bt, Hkv, L, D), generator=g, device="cuda", dtype=torch.bfloat16)
    p = laq.params_for(q, k, W, 7, 100)
    p.group_mode = group
    ws = laq.alloc_workspace(p, "cuda")
    scores = torch.zeros((NL, Bt, Hkv * (G if group == 2 else 1), L - W), device="cuda")
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)

    def run():
        scores.zero_()
        assert hooked.laq_score(ctypes.byref(p), q.data_ptr(), k.data_ptr(), scores.data_ptr(), ws.data_ptr(),
                                ws.numel(), stream) == laq.LAQ_OK
        assert hooked.laq_test_last_cluster() == C
        return hooked.laq_last_device_status(ctypes.byref(p), ws.data_ptr(), ws.numel(), stream)

    assert run() == laq.LAQ_OK
    want = scores.clone()
    hooked.laq_test_withhold_unit(1)
    try:
        assert run() == laq.LAQ_ERR_TIMEOUT
    finally:
        hooked.laq_test_withhold_unit(-1)
    assert run() == laq.LAQ_OK
    assert torch.equal(scores, want)


def test_wait_that_runs_out_where_tiles_are_handed_over_whole():
    # 200 units of 160 rows and five tiles: more than two tasks an SM, short ones
    from paper_2505_20334_b200 import binding as laq

    hooked = hooked_library()
    Bt, G, Hkv, W, D, L = 100, 5, 2, 32, 128, 600
    g = torch.Generator(device="cuda").manual_seed(7)
    q = torch.randn((1, Bt, G * Hkv, W, D), generator=g, device="cuda", dtype=torch.bfloat16)
    k = torch.randn((1, Bt, Hkv, L, D), generator=g, device="cuda", dtype=torch.bfloat16)
    p = laq.params_for(q, k, W, 7, 100)
    ws = laq.alloc_workspace(p, "cuda")
    scores = torch.zeros((1, Bt, Hkv, L - W), device="cuda")
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)

    def run(lib):
        scores.zero_()
        assert lib.laq_score(ctypes.byref(p), q.data_ptr(), k.data_ptr(), scores.data_ptr(), ws.data_ptr(), ws.numel(),
                             stream) == laq.LAQ_OK
        return lib.laq_last_device_status(ctypes.byref(p), ws.data_ptr(), ws.numel(), stream)

    assert run(hooked) == laq.LAQ_OK
    want = scores.clone()
    for unit in (0, 1, 150, 199):
        hooked.laq_test_withhold_unit(unit)
        try:
            assert run(hooked) == laq.LAQ_ERR_TIMEOUT
        finally:
            hooked.laq_test_withhold_unit(-1)
    for lib in (hooked, laq.lib):
        assert run(lib) == laq.LAQ_OK
        assert float((scores - want).norm() / want.norm()) < 5e-7     # (tasks of an odd number of tiles)
