"""laq_evict_host on caches large enough to be taken in pieces of layers: copies on a second stream,
scoring and gather behind them. Kept sets against the device run (equal but for scores that tie with
the last kept one to fp32 rounding), rows bit for bit."""
import numpy as np
import pytest
import torch

from parity_util import bits
from test_gpu_parity import laq, rand_inputs  # noqa: F401 (laq is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pinned", [True, False])
@pytest.mark.parametrize("lens", [None, (4100, 3001)])
def test_host_cache_in_pieces_equals_device_run(laq, pinned, lens):
    NL, Bt, Hq, Hkv, D, L, W, kernel, B = 5, 2, 4, 2, 128, 4100, 8, 7, 200   # 21 MB of keys
    q, k, v = rand_inputs(NL, Bt, Hq, Hkv, D, L, W, seed=41, kscale=1.5)
    dev = laq.evict(q.cuda(), k.cuda(), v.cuda(), B, pool_kernel=kernel, seq_lens=lens, want_scores=True)
    scores, want = dev["scores"].cpu().numpy(), dev["idx"].cpu().numpy()
    he = laq.HostEvictor(tuple(q.shape), tuple(k.shape), B, kernel, W, "cuda")
    he.params.set_seq_lens(lens)
    host = [t.pin_memory() if pinned else t.clone() for t in (q, k, v)]
    side = torch.cuda.Stream()
    for stream in (None, side, None):       # calls in a row share staging and the second stream
        he.h_k_out.zero_(); he.h_v_out.zero_(); he.h_idx.zero_()
        torch.cuda.synchronize()
        hk, hv, hidx = he.run(*host, stream=stream)
        torch.cuda.synchronize()
        assert laq.laq_last_device_status(he.params, he.ws) == laq.LAQ_OK
        got = hidx.numpy()
        for n in range(NL):
            for b in range(Bt):
                for h in range(Hkv):
                    a, w, s = got[n, b, h], want[n, b, h], scores[n, b, h]
                    theta = s[w[:B - W]].min()
                    diff = np.array(sorted(set(a.tolist()) ^ set(w.tolist())), dtype=np.int64)
                    assert (np.abs(s[diff] - theta) <= 1e-5 * theta).all()
                    assert (bits(hk[n, b, h]) == bits(k[n, b, h])[a]).all()
                    assert (bits(hv[n, b, h]) == bits(v[n, b, h])[a]).all()


def test_host_call_while_another_one_is_being_captured(laq):
    # The copies of a large host cache run on a second stream, which a capture of the caller's stream takes
    # in. A call on another stream meanwhile must neither join that capture nor fail.
    NL, Bt, Hq, Hkv, D, L, W, kernel, B = 4, 1, 4, 2, 128, 4100, 8, 7, 200   # 8.4 MB of keys: two pieces
    sets = [[t.pin_memory() for t in rand_inputs(NL, Bt, Hq, Hkv, D, L, W, seed=s, kscale=1.5)] for s in (1, 2)]
    evictors = [laq.HostEvictor(tuple(q.shape), tuple(k.shape), B, kernel, W, "cuda") for q, k, _ in sets]
    want = []
    for he, host in zip(evictors, sets):
        he.run(*host)
        torch.cuda.synchronize()
        want.append([t.clone() for t in (he.h_k_out, he.h_v_out, he.h_idx)])
        for t in (he.h_k_out, he.h_v_out, he.h_idx):
            t.zero_()
    capturing, other = torch.cuda.Stream(), torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=capturing, capture_error_mode="relaxed"):
        evictors[0].run(*sets[0], stream=capturing)
        evictors[1].run(*sets[1], stream=other)
        evictors[0].run(*sets[0], stream=capturing)
    other.synchronize()
    assert not evictors[0].h_idx.any()                     # captured, not run
    for _ in range(2):
        graph.replay()
        torch.cuda.synchronize()
        for he, w in zip(evictors, want):
            for got, ref in zip((he.h_k_out, he.h_v_out, he.h_idx), w):
                assert torch.equal(got.view(torch.int16), ref.view(torch.int16))
    evictors[0].run(*sets[0])                              # and the second stream works as before
    torch.cuda.synchronize()
    assert torch.equal(evictors[0].h_idx, want[0][2])


def test_stage_events_of_a_host_call_span_all_its_pieces(laq):
    # 32 MB of keys in pieces: the copy of the last pieces lies between the first scoring and the last
    NL, Bt, Hq, Hkv, D, L, W, kernel, B = 8, 1, 4, 2, 128, 8192, 8, 7, 200
    host = [t.pin_memory() for t in rand_inputs(NL, Bt, Hq, Hkv, D, L, W, seed=3)]
    he = laq.HostEvictor(tuple(host[0].shape), tuple(host[1].shape), B, kernel, W, "cuda")
    events = [torch.cuda.Event(enable_timing=True) for _ in range(4)]
    for e in events:
        e.record()
    he.run(*host)
    torch.cuda.synchronize()
    laq.laq_set_stage_events(events[1], events[2])
    try:
        events[0].record()
        he.run(*host)
        events[3].record()
    finally:
        laq.laq_set_stage_events()
    torch.cuda.synchronize()
    # eight pieces: from the first one's scoring to the last one's is most of the call
    assert events[1].elapsed_time(events[2]) > 0.5 * events[0].elapsed_time(events[3])
