"""Inverse-CDF sampling with many rays per warp, against the FP64 oracle: ray counts around the groups'
edges, sample counts that are no multiple of a warp, one bin, bins spread unevenly over the lanes, probability
mass in single bins, runs of zero bins across lane borders, rays that miss the box; every dt equals the
difference of its neighbours' t to an FP32 ulp of t."""
import numpy as np
import pytest
import torch

import oracle
import synth
from test_gpu_parity import cuda

pytestmark = pytest.mark.gpu

dvgo = pytest.importorskip("paper_2111_11215_gb300")


@pytest.mark.parametrize("R,nb,ns,eta", [(1, 64, 33, 0.0), (31, 1, 5, 0.05), (1217, 64, 48, 0.0), (2433, 33, 31, 0.01),
                                         (1300, 128, 65, 0.0), (1300, 97, 1, 0.0)])
def test_sample_pdf_groups_match_oracle(R, nb, ns, eta):
    g = np.random.default_rng(R + nb)
    o, d, jit, _ = synth.fine_batch(R, 3)
    o[::7] += 9.0                                                 # some rays miss the box
    probs = g.uniform(size=(R, nb)) ** 6
    probs[R // 3::3] *= g.uniform(size=(len(probs[R // 3::3]), nb)) < 0.3      # zero bins, also whole lanes of them
    probs[:, nb // 2] += 1e-3
    spike = np.arange(0, R, 5)
    probs[spike] = 0.0
    probs[spike, g.integers(0, nb, len(spike))] = 1.0
    probs = (probs / probs.sum(1, keepdims=True)).astype(np.float32)
    p = dvgo.Params(mode=dvgo.DVGO_MODE_FINE, step=0.01)
    dd = dvgo.GridDesc((16,) * 3, 1)
    t, dt = torch.full((R, ns), -1.0, device="cuda"), torch.full((R, ns), -1.0, device="cuda")
    dvgo.dvgo_sample_pdf(p, dd, cuda(o), cuda(d), cuda(probs), ns, cuda(jit), eta, t, dt)
    torch.cuda.synchronize()
    t, dt = t.cpu().numpy(), dt.cpu().numpy()
    P = oracle.Params(grid_shape=(16,) * 3, shift_b=0.0, delta=0.01, bg=(1.0, 1.0, 1.0), mode=1, feat_dim=12, n_freq=4,
                      hidden=128)
    e = float(np.float32(eta))
    for r in range(0, R, max(1, R // 200)):
        _, t0, t1, _, _ = oracle.ray_bounds(P, o[r], d[r], 0.5)
        if t1 <= t0:
            assert not t[r].any() and not dt[r].any()
            continue
        tr, dtr = oracle.sample_pdf(probs[r].astype(np.float64), t0, t1, ns, jit=float(jit[r]), eta=e)
        np.testing.assert_allclose(t[r], tr, rtol=2 ** -22)
        np.testing.assert_allclose(dt[r], dtr, rtol=1e-5, atol=2 ** -22 * t1)
