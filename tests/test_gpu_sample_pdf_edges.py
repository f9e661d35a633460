"""Inverse-CDF sampling at the edges of its inputs: a jitter outside [0, 1) extrapolates the first and the last bin, a
NaN probability or a ray without any probability gives NaN (not a finite distance), and ordinary rays of the same
batch are untouched.  Distances against the FP64 formula, to FP32 rounding (2^-22)."""
import numpy as np
import pytest
import torch

import oracle
import synth
from test_gpu_parity import cuda

pytestmark = pytest.mark.gpu

dvgo = pytest.importorskip("paper_2111_11215_gb300")

R, NB, NS = 65, 64, 40


def test_sample_pdf_edges():
    g = np.random.default_rng(95)
    o, d, _, _ = synth.fine_batch(4 * R, 96)
    P = oracle.Params(grid_shape=(16,) * 3, shift_b=0.0, delta=0.01, bg=(1.0, 1.0, 1.0), mode=1, feat_dim=12, n_freq=4,
                      hidden=128)
    bounds = [oracle.ray_bounds(P, o[r], d[r], 0.5)[1:3] for r in range(4 * R)]
    hit = [r for r in range(4 * R) if bounds[r][1] > bounds[r][0]][:R]
    assert len(hit) == R
    o, d = o[hit], d[hit]
    probs = g.uniform(0.2, 1.0, size=(R, NB))
    probs = (probs / probs.sum(1, keepdims=True)).astype(np.float32)
    jit = g.uniform(size=R).astype(np.float32)
    jit[::4], jit[1::4] = -0.75, 1.6
    probs[2, 0], probs[2, 20] = 0.0, np.nan
    probs[6] = 0.0
    t, dt = torch.empty((R, NS), device="cuda"), torch.empty((R, NS), device="cuda")
    dvgo.dvgo_sample_pdf(dvgo.Params(mode=dvgo.DVGO_MODE_FINE, step=0.01), dvgo.GridDesc((16,) * 3, 1), cuda(o), cuda(d),
                         cuda(probs), NS, cuda(jit), 0.0, t, dt)
    torch.cuda.synchronize()
    t = t.cpu().numpy()
    assert np.isnan(t[2]).all() and np.isnan(t[6]).all()
    for r in set(range(R)) - {2, 6}:
        t0, t1 = bounds[hit[r]]
        q = probs[r].astype(np.float64)
        Q = np.concatenate([[0.0], np.cumsum(q)])
        u = (np.arange(NS) + float(jit[r])) / NS * Q[-1]
        b = np.clip(np.searchsorted(Q[1:], u, side="right"), 0, NB - 1)
        ref = t0 + (b + (u - Q[b]) / q[b]) * (t1 - t0) / NB
        np.testing.assert_allclose(t[r], ref, rtol=2 ** -22, err_msg=str(r))
