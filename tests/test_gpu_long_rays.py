"""Rays of more than 1024 samples (up to 2048 are accepted), whose kept samples fill more than 32 chunks of 32: forward,
backward and labels against the FP64 oracle, with every sample kept, with known gaps (whole chunks of removed samples
at the front, in the middle and at the end) and with rays that terminate late.  Tolerances as everywhere for the FP32
path: 1e-5 on colours and labels, the oracle's running error bound on gradients."""
import numpy as np
import pytest
import torch

import oracle
import synth
from helpers import BOUND_FP32, RTOL_COLOUR, assert_close, mlp_flat, oracle_params
from test_gpu_bf16_tiles import _check
from test_gpu_fine_edges import RES, _hitting_rays
from test_gpu_parity import _fine_inputs

pytestmark = pytest.mark.gpu

dvgo = pytest.importorskip("paper_2111_11215_gb300")

R = 9


@pytest.mark.parametrize("kind", ["all", "gaps", "late"])
def test_long_rays_match_oracle(kind, capsys):
    _, feat, _, _, _, _, _ = _fine_inputs(RES, 8, seed=890)
    mlp = synth.mlp_weights(39, 128, 3, 893)
    g = np.random.default_rng(891)
    dens = g.normal(scale=0.3, size=(RES,) * 3).astype(np.float32)
    x = np.linspace(-1, 1, RES)
    if kind == "gaps":
        dens[(np.abs(x) > 0.7) | (np.abs(x) < 0.25)] = -60.0
    if kind == "late":
        dens[x > 0.5] = 4000.0
    o, d, t0, t1 = _hitting_rays(400, 892)
    long = np.nonzero(t1 - t0 > 2.1)[0][:R]
    assert len(long) == R
    o, d = o[long], d[long]
    p = dvgo.Params(mode=dvgo.DVGO_MODE_FINE, step=0.0018, bg=(0.25, 0.5, 0.75), shift_b=-1.0,
                    tau_f=1e-6 if kind == "gaps" else 0.0, mlp_prec=dvgo.DVGO_MLP_FP32)
    gC = g.normal(scale=1e-2, size=(R, 3))
    dd, cd = dvgo.GridDesc((RES,) * 3, 1), dvgo.GridDesc((RES,) * 3, 12)
    cu = lambda a: torch.as_tensor(np.ascontiguousarray(a)).to(device="cuda", dtype=torch.float32)  # noqa: E731
    D, F, flat = cu(dens), cu(feat), cu(mlp_flat(mlp))
    views = dvgo.render.mlp_views(flat, 39)
    r = dvgo.Renderer(p, dd, cd, R)
    rgb, tf, _ = r.forward(D, F, views, cu(o), cu(d), None)
    labels = torch.empty((R, 64), device="cuda")
    dvgo.dvgo_weight_bins(p, dd, R, 64, r.workspace, labels)
    g_d, g_f, g_m = torch.zeros_like(D), torch.zeros_like(F), torch.zeros_like(flat)
    r.backward(D, F, views, cu(o), cu(d), None, None, cu(gC), None, g_d, g_f, g_m)
    torch.cuda.synchronize()
    kept = int(r.workspace[8:12].view(torch.int32).item())
    assert kept > R * {"all": 1100, "gaps": 300, "late": 200}[kind]
    ref = oracle.render(oracle_params(p, (RES,) * 3, 12), dens, feat, o, d, mlp=mlp, grad_rgb=gC, n_bins=64,
                        error_bound=BOUND_FP32)
    assert_close(rgb.cpu().numpy(), ref.rgb, RTOL_COLOUR, "rgb")
    assert_close(tf.cpu().numpy(), ref.tfinal, RTOL_COLOUR, "tfinal")
    assert_close(labels.cpu().numpy(), ref.wbins, RTOL_COLOUR, "labels")
    got = {"rgb": rgb.cpu().numpy(), "g_d": g_d.reshape((RES,) * 3).cpu().numpy(),
           "g_f": g_f.reshape((RES,) * 3 + (12,)).cpu().numpy(), "g_m": g_m.cpu().numpy()}
    _check(got, ref, capsys, f"long rays, {kind}: {kept} kept")
