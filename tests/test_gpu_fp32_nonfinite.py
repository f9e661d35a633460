"""Infinite and huge features and weights in the FP32 colour forward: the colours are what FP32 arithmetic gives (NaN, a
saturated sigmoid, or a number where a sum of both infinities makes a hidden unit NaN), and samples
without them are untouched.  One sample a ray, ragged tiles, 39 and 72 inputs, both layouts; against an FP64
evaluation with ReLU(NaN) = 0, whose infinities and NaN are the same."""
import numpy as np
import pytest
import torch

import synth
from helpers import RTOL_COLOUR
from test_gpu_fine_edges import RES, _explicit_samples, _hitting_rays, _params
from test_gpu_parity import _mlp_flat, cuda

pytestmark = pytest.mark.gpu

dvgo = pytest.importorskip("paper_2111_11215_gb300")

R = 300


def _colours(feat, mlp, o, d, ts, pe_x):
    e = d.astype(np.float64) / np.linalg.norm(d.astype(np.float64), axis=1, keepdims=True)
    x = o.astype(np.float64) + ts.astype(np.float64) * e
    u = (x + 1.0) * (RES - 1) / 2.0
    i0 = np.clip(np.floor(u), 0, RES - 2).astype(int)
    f = (u - i0).astype(np.float32).astype(np.float64)
    v = np.zeros((len(o), 12))
    for q in range(8):
        b = np.array([q >> 2 & 1, q >> 1 & 1, q & 1])
        w = np.where(b, f, 1.0 - f).prod(1)
        i = i0 + b
        v += w[:, None] * feat[i[:, 0], i[:, 1], i[:, 2]].astype(np.float64)

    def pe(x, n):
        a = x[:, :, None] * 2.0 ** np.arange(n)
        return np.concatenate([x, np.sin(a).reshape(len(x), -1), np.cos(a).reshape(len(x), -1)], 1)

    h = np.concatenate([v, pe(e, 4)] + ([pe(x, 5)] if pe_x else []), 1)
    for i in ("1", "2"):
        z = (h[:, :, None] * mlp["w" + i].astype(np.float64)).sum(1) + mlp["b" + i]
        h = np.where(z > 0, z, 0.0)
    z = (h[:, :, None] * mlp["w3"].astype(np.float64).reshape(128, 3)).sum(1) + mlp["b3"]
    return 1.0 / (1.0 + np.exp(-z))


@pytest.mark.parametrize("pe_x,packed", [(0, 0), (5, 0), (0, 1)])
@pytest.mark.parametrize("kind", ["feature", "huge", "weight1", "weight2"])
def test_infinities_go_through_as_fp32(pe_x, packed, kind):
    g = np.random.default_rng(885)
    dens = np.full((RES,) * 3, 60.0, np.float32)
    feat = g.normal(size=(RES,) * 3 + (12,)).astype(np.float32)
    mlp = synth.mlp_weights(72 if pe_x else 39, 128, 3, 886)
    o, d, t0, t1 = _hitting_rays(R, 887)
    ts, _ = _explicit_samples(t0, t1, 1, 888)
    dts = np.full_like(ts, 0.5)
    if kind == "feature":
        at = g.integers(0, RES, size=(60, 3))
        feat[at[:, 0], at[:, 1], at[:, 2], g.integers(0, 12, 60)] = np.where(g.uniform(size=60) < 0.5, np.inf, -np.inf)
        mlp["w1"][:4] = np.abs(mlp["w1"][:4])               # one sign: some sums keep their infinity
        mlp["w2"] = np.where(np.arange(128)[None, :] < 3, np.abs(mlp["w2"]), mlp["w2"]).astype(np.float32)
        mlp["w3"][3:] = 0.0
    if kind == "huge":
        feat[::2] *= 1e37
        mlp["w1"][:12] *= 1e-30
    if kind == "weight1":
        mlp["w1"][5, 7] = np.inf
    if kind == "weight2":
        mlp["w2"][9, 3] = -np.inf
    p = _params(dvgo.DVGO_MLP_FP32, n_freq_pos=pe_x)
    dd, cd = dvgo.GridDesc((RES,) * 3, 1), dvgo.GridDesc((RES,) * 3, 12)
    D, F = cuda(dens), cuda(feat)
    if packed:
        D, F = dvgo.dvgo_pack_grid(dd, D, dd.with_(layout=1)), dvgo.dvgo_pack_grid(cd, F, cd.with_(layout=1))
        dd, cd = dd.with_(layout=1), cd.with_(layout=1)
    r = dvgo.Renderer(p, dd, cd, R, samples_per_ray=1)
    views = dvgo.render.mlp_views(cuda(_mlp_flat(mlp)), 72 if pe_x else 39)
    rgb, tf, _ = r.forward(D, F, views, cuda(o), cuda(d), None, (cuda(ts), cuda(dts)))
    torch.cuda.synchronize()
    assert dvgo.dvgo_workspace_status(r.workspace) == 0
    T = np.exp(-(60.0 + p.shift_b) * 0.5)                   # softplus(z) = z there
    assert T < 1e-6
    with np.errstate(all="ignore"):
        c = _colours(feat, mlp, o, d, ts, pe_x)
    got = rgb.cpu().numpy().astype(np.float64)
    assert np.array_equal(np.isnan(got), np.isnan(c)), (np.isnan(got).sum(), np.isnan(c).sum())
    ok = ~np.isnan(c)
    np.testing.assert_allclose(got[ok], c[ok], rtol=RTOL_COLOUR, atol=RTOL_COLOUR)
