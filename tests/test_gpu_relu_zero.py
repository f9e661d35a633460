"""Hidden units whose pre-activation is exactly 0 (incoming weights and bias all 0, as after zero
initialisation or pruning) are off in the FP32 colour backward, as in the oracle ([z > 0]): both layers, 39 and
72 inputs, and the whole first layer at 0 with a bias of 0 behind it.  Tolerances as everywhere for the FP32
path, against the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth
from helpers import BOUND_FP32, RTOL_COLOUR, assert_close, mlp_flat, oracle_params
from test_gpu_bf16_tiles import _check
from test_gpu_fine_edges import RES, _explicit_samples, _hitting_rays, _params
from test_gpu_parity import _fine_inputs

pytestmark = pytest.mark.gpu

dvgo = pytest.importorskip("paper_2111_11215_gb300")

R, K = 37, 16


@pytest.mark.parametrize("pe_x,whole", [(0, False), (5, False), (0, True)])
def test_zero_units_pass_no_gradient(pe_x, whole, capsys):
    dens, feat, _, _, _, _, _ = _fine_inputs(RES, 8, seed=870)
    mlp = synth.mlp_weights(72 if pe_x else 39, 128, 3, 871)
    one, two = ([3, 64, 77], [5, 100]) if not whole else (list(range(128)), [0, 99])
    mlp["w1"][:, one], mlp["b1"][one] = 0.0, 0.0
    mlp["b2"][two] = 0.0
    if not whole:
        mlp["w2"][:, two] = 0.0
    o, d, t0, t1 = _hitting_rays(R, 872)
    ts, dts = _explicit_samples(t0, t1, K, 873)
    p = _params(dvgo.DVGO_MLP_FP32, n_freq_pos=pe_x)
    gC = np.random.default_rng(874).normal(scale=1e-2, size=(R, 3))
    dd, cd = dvgo.GridDesc((RES,) * 3, 1), dvgo.GridDesc((RES,) * 3, 12)
    cu = lambda a: torch.as_tensor(np.ascontiguousarray(a)).to(device="cuda", dtype=torch.float32)  # noqa: E731
    D, F, flat = cu(dens), cu(feat), cu(mlp_flat(mlp))
    views = dvgo.render.mlp_views(flat, 72 if pe_x else 39)
    r = dvgo.Renderer(p, dd, cd, R, samples_per_ray=K)
    samples = (cu(ts), cu(dts))
    rgb, _, _ = r.forward(D, F, views, cu(o), cu(d), None, samples)
    g_d, g_f, g_m = torch.zeros_like(D), torch.zeros_like(F), torch.zeros_like(flat)
    r.backward(D, F, views, cu(o), cu(d), None, samples, cu(gC), None, g_d, g_f, g_m)
    torch.cuda.synchronize()
    ref = oracle.render(oracle_params(p, (RES,) * 3, 12), dens, feat, o, d, mlp=mlp, explicit_t=ts, explicit_dt=dts,
                        grad_rgb=gC, error_bound=BOUND_FP32)
    assert_close(rgb.cpu().numpy(), ref.rgb, RTOL_COLOUR, "rgb")
    got = {"rgb": rgb.cpu().numpy(), "g_d": g_d.reshape((RES,) * 3).cpu().numpy(),
           "g_f": g_f.reshape((RES,) * 3 + (12,)).cpu().numpy(), "g_m": g_m.cpu().numpy()}
    _check(got, ref, capsys, f"zero units, pe_x {pe_x}, whole {whole}")
    g = dvgo.render.mlp_views(g_m, 72 if pe_x else 39)
    for k, cols in (("w1", one), ("b1", one), ("b2", two)):
        assert not g[k].reshape(-1, 128)[:, cols].any(), k


def test_nan_feature_turns_its_units_off():
    """A NaN feature makes every unit of the first layer NaN: off, as [z > 0] is.  The lattice points that only samples
    with a NaN corner touch get a feature gradient of exactly 0, and b1, w2, b2, w3, b3 gradients stay finite."""
    dens, feat, mlp, _, _, _, _ = _fine_inputs(RES, 8, seed=875)
    feat[10:13, 10:13, 10:13] = np.nan
    o, d, t0, t1 = _hitting_rays(R, 876)
    ts, dts = _explicit_samples(t0, t1, K, 877)
    ts[0], dts[0] = np.linspace(3.9, 3.95, K), 0.003             # through the middle of the NaN block
    e = np.array([0.11, 0.23, 0.97])
    o[0], d[0] = -3.93 * e / np.linalg.norm(e), e / np.linalg.norm(e)
    cu = lambda a: torch.as_tensor(np.ascontiguousarray(a)).to(device="cuda", dtype=torch.float32)  # noqa: E731
    D, F, flat = cu(dens), cu(feat), cu(mlp_flat(mlp))
    p = _params(dvgo.DVGO_MLP_FP32)
    r = dvgo.Renderer(p, dvgo.GridDesc((RES,) * 3, 1), dvgo.GridDesc((RES,) * 3, 12), R, samples_per_ray=K)
    views, samples = dvgo.render.mlp_views(flat, 39), (cu(ts), cu(dts))
    rgb, _, _ = r.forward(D, F, views, cu(o), cu(d), None, samples)
    assert torch.isfinite(rgb).all()
    g_d, g_f, g_m = torch.zeros_like(D), torch.zeros(F.shape, device="cuda"), torch.zeros_like(flat)
    gC = cu(np.random.default_rng(878).normal(scale=1e-2, size=(R, 3)))
    r.backward(D, F, views, cu(o), cu(d), None, samples, gC, None, g_d, g_f, g_m)
    torch.cuda.synchronize()
    g = dvgo.render.mlp_views(g_m, 39)
    assert torch.isnan(g["w1"][:12]).any() and all(torch.isfinite(g[k]).all() for k in ("b1", "w2", "b2", "w3", "b3"))
    g_f = g_f.reshape((RES,) * 3 + (12,))
    assert torch.isfinite(g_f).all() and not g_f[11, 11, 11].any() and g_f.any()
