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
