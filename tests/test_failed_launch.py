"""A launch that CUDA refuses is reported by the call that made it and by no later one."""
import ctypes

import pytest
import torch

from test_gpu_parity import laq, rand_inputs  # noqa: F401 (laq is a fixture)

pytestmark = pytest.mark.gpu


def test_a_refused_launch_leaves_no_error_behind(laq):  # noqa: F811
    # A stream whose capture has been invalidated (by a synchronise while it captures) refuses launches:
    # an error on the host only, over when the capture ends.
    q, k, v = (t.cuda() for t in rand_inputs(1, 1, 8, 2, 128, 600, 8, seed=2))
    wide = rand_inputs(1, 1, 8, 2, 128, 600, 32, seed=3)[0].cuda()      # 128 rows
    B = 60
    calls = {}
    for name, queries, opts in (("cluster", q, {}), ("two sweeps", wide, {}), ("raw", q, {"score_mode": 1})):
        out = laq.evict(queries, k, v, B, want_scores=True, **opts)
        calls[name] = (out, queries)
    rt = ctypes.CDLL("libcudart.so.12")
    side = torch.cuda.Stream()
    raw = ctypes.c_void_p(side.cuda_stream)
    idx = calls["cluster"][0]["idx"]

    def in_broken_capture(call):
        torch.cuda.synchronize()
        assert rt.cudaStreamBeginCapture(raw, 2) == 0            # relaxed: other threads stay unaffected
        assert rt.cudaStreamSynchronize(raw) != 0                # not allowed while capturing
        try:
            return call()
        finally:
            graph = ctypes.c_void_p()
            assert rt.cudaStreamEndCapture(raw, ctypes.byref(graph)) != 0
            rt.cudaGetLastError()

    def later_calls_work():
        for out, queries in calls.values():
            scores = torch.empty_like(out["scores"])
            assert laq.laq_score(out["params"], queries, k, scores, out["ws"], check=False) == laq.LAQ_OK
            assert torch.equal(scores, out["scores"])

    common = torch.empty(2, dtype=torch.int32, device="cuda")
    for out, queries in calls.values():
        p, ws = out["params"], out["ws"]
        assert in_broken_capture(lambda: laq.laq_evict(
            p, queries, k, v, out["k_out"], out["v_out"], out["idx"], None, ws, side, check=False)) == laq.LAQ_ERR_CUDA
        later_calls_work()
    p = calls["cluster"][0]["params"]
    for call in (lambda: laq.laq_select(p, calls["cluster"][0]["scores"], idx, side, check=False),
                 lambda: laq.laq_compact(p, k, v, idx, calls["raw"][0]["k_out"], None, side, check=False),
                 lambda: laq.lib.laq_recall(2, idx.data_ptr(), B, idx.data_ptr(), B, common.data_ptr(), None,
                                            side.cuda_stream)):
        assert in_broken_capture(call) == laq.LAQ_ERR_CUDA
        later_calls_work()
