"""Labels from a workspace that was rendered with other parameters than the labels' call has: another step (the bins are
then those of the call's step), explicit samples, more rays.  The state is found where the forward left it.  The
same weights summed in other bins or in another order: FP32 rounding of sums of at most 90 terms (90 x 2^-24)."""
import numpy as np
import pytest
import torch

import synth
from test_gpu_parity import _mlp_flat, cuda

pytestmark = pytest.mark.gpu

dvgo = pytest.importorskip("paper_2111_11215_gb300")

RES, R, STEP = 24, 300, 0.045
TOL = 90 * 2 ** -24


def _setup():
    g = np.random.default_rng(71)
    dens = cuda((g.normal(size=(RES,) * 3) * 2.0).astype(np.float32))
    feat = cuda(g.normal(size=(RES,) * 3 + (12,)).astype(np.float32))
    flat = cuda(_mlp_flat(synth.mlp_weights(39, 128, 3, 72)))
    o, d, _, _ = (cuda(a) for a in synth.fine_batch(R, 73))
    p = dvgo.Params(mode=dvgo.DVGO_MODE_FINE, step=STEP, shift_b=-1.0, tau_f=1e-2)
    dd, cd = dvgo.GridDesc((RES,) * 3, 1), dvgo.GridDesc((RES,) * 3, 12)
    r = dvgo.Renderer(p, dd, cd, R)
    r.forward(dens, feat, dvgo.mlp_views(flat), o, d)
    return p, dd, cd, r, (dens, feat, dvgo.mlp_views(flat), o, d)


def _labels(p, dd, n, bins, ws):
    out = torch.full((n, bins), float("nan"), device="cuda")
    dvgo.dvgo_weight_bins(p, dd, n, bins, ws, out)
    torch.cuda.synchronize()
    return out


def test_another_step():
    """64 bins at twice the step: sample k falls where it does in 128 bins at the step, the last bin taking the rest."""
    p, dd, _, r, _ = _setup()
    fine = _labels(p, dd, R, 128, r.workspace)
    got = _labels(p.with_(step=2 * STEP), dd, R, 64, r.workspace)
    hit = (fine - 1 / 128).abs().amax(1) > 1e-3
    assert hit.sum() > R // 3
    torch.testing.assert_close(got[hit, :63], fine[hit, :63], rtol=TOL, atol=TOL)
    torch.testing.assert_close(got[hit, 63], fine[hit, 63:].sum(1), rtol=TOL, atol=TOL)


def test_fewer_rays():
    p, dd, _, r, _ = _setup()
    torch.testing.assert_close(_labels(p, dd, R // 2, 64, r.workspace), _labels(p, dd, R, 64, r.workspace)[:R // 2],
                               rtol=TOL, atol=TOL)


def test_explicit_samples():
    """Explicit samples at the uniform ones' places (and steps of 0 where a ray has no more): the same labels."""
    p, dd, cd, r, args = _setup()
    counts = torch.empty(R, dtype=torch.int32, device="cuda")
    dvgo.dvgo_sample_counts(r.workspace, R, counts)
    ref = _labels(p, dd, R, 64, r.workspace)
    k = torch.arange(90, device="cuda")
    assert int(counts.max()) <= 90
    o, d = args[3].double(), args[4].double()
    e = d / d.norm(dim=1, keepdim=True)
    t1, t2 = (-1.0 - o) / e, (1.0 - o) / e
    t0 = torch.minimum(t1, t2).amax(1).clamp(min=0.0)
    t = (t0[:, None] + (k + 0.5) * STEP).float()
    dt = torch.where(k < counts[:, None], torch.tensor(STEP, device="cuda"), torch.tensor(0.0, device="cuda"))
    x = dvgo.Renderer(p, dd, cd, R, samples_per_ray=90)
    x.forward(*args, None, (t.contiguous(), dt.contiguous()))
    got = _labels(p, dd, R, 64, x.workspace)
    # (t is rounded to FP32: 2^-24 x 5 in x, densities that change by up to 10 a cell of 0.09, weights of at most 1; and
    # a sample whose alpha that takes across tau_f moves weights by 1e-2)
    near = (got - ref).abs().amax(1) < 1e-3
    assert near.sum() >= R - 3, int((~near).sum())
