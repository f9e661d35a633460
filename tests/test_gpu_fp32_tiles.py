"""The FP32 colour kernels at the edges of their 128-row tiles, against the FP64 oracle: one sample, one
below, at and above a tile, exactly two tiles for every CTA, and a ragged third, with explicit samples that
are all kept; 39 and 72 inputs, FP32 and BF16 features, both layouts.  Also weights and features of very
different sizes, whose three-way BF16 split must stay exact to FP32.  Tolerances as everywhere for
the FP32 path: 1e-5 on colours, 1e-4 (plus the oracle's running error bound) on gradients."""
import numpy as np
import pytest
import torch

import oracle
import synth
from helpers import BOUND_FP32, RTOL_COLOUR, assert_close, mlp_flat, oracle_params
from test_gpu_bf16_tiles import _bf16, _check
from test_gpu_fine_edges import RES, _explicit_samples, _hitting_rays, _params
from test_gpu_parity import _fine_inputs

pytestmark = pytest.mark.gpu

dvgo = pytest.importorskip("paper_2111_11215_gb300")

_RAYS = {}


def _rays(R, K):
    if (R, K) not in _RAYS:
        o, d, t0, t1 = _hitting_rays(R, 831)
        _RAYS[R, K] = (o, d) + _explicit_samples(t0, t1, K, 832)
    return _RAYS[R, K]


@pytest.mark.parametrize("R,K,pe_x,bf16_feat,packed,scale", [
    (1, 1, 0, False, 0, 1.0), (127, 1, 5, True, 0, 1.0), (128, 1, 0, False, 1, 1.0), (129, 1, 5, False, 0, 1.0),
    (608, 64, 0, False, 0, 1.0), (611, 64, 5, False, 1, 1.0), (611, 64, 0, True, 0, 1.0),
    (37, 48, 0, False, 0, 1e3), (37, 48, 5, False, 0, 1e-3),
])
def test_fp32_tiles_match_oracle(R, K, pe_x, bf16_feat, packed, scale, capsys):
    dens, feat, _, _, _, _, _ = _fine_inputs(RES, 8, seed=830)
    mlp = synth.mlp_weights(72 if pe_x else 39, 128, 3, 833)
    # features and first-layer rows of very different sizes whose products stay ordinary
    feat = (feat * scale).astype(np.float32)
    mlp["w1"][:12] = (mlp["w1"][:12] / scale).astype(np.float32)
    if bf16_feat:
        feat = _bf16(feat)
    o, d, ts, dts = _rays(R, K)
    p = _params(dvgo.DVGO_MLP_FP32, n_freq_pos=pe_x)
    gC = np.random.default_rng(834).normal(scale=1e-2, size=(R, 3))
    dt = torch.bfloat16 if bf16_feat else torch.float32
    dd = dvgo.GridDesc((RES,) * 3, 1)
    cd = dvgo.GridDesc((RES,) * 3, 12, dtype=dvgo.DVGO_DTYPE_BF16 if bf16_feat else dvgo.DVGO_DTYPE_F32)
    cu = lambda a, t=torch.float32: torch.as_tensor(np.ascontiguousarray(a)).to(device="cuda", dtype=t)  # noqa: E731
    D, F, flat = cu(dens), cu(feat, dt), cu(mlp_flat(mlp))
    if packed:
        D, F = dvgo.dvgo_pack_grid(dd, D, dd.with_(layout=1)), dvgo.dvgo_pack_grid(cd, F, cd.with_(layout=1))
        dd, cd = dd.with_(layout=1), cd.with_(layout=1)
    views = dvgo.render.mlp_views(flat, 72 if pe_x else 39)
    r = dvgo.Renderer(p, dd, cd, R, samples_per_ray=K)
    samples = (cu(ts), cu(dts))
    rgb, tf, _ = r.forward(D, F, views, cu(o), cu(d), None, samples)
    g_d, g_f, g_m = torch.zeros_like(D), torch.zeros(F.shape, device="cuda"), torch.zeros_like(flat)
    r.backward(D, F, views, cu(o), cu(d), None, samples, cu(gC), None, g_d, g_f, g_m)
    if packed:
        g_d = dvgo.dvgo_pack_grid(dd, g_d, dd.with_(layout=0))
        c32 = cd.with_(dtype=dvgo.DVGO_DTYPE_F32)
        g_f = dvgo.dvgo_pack_grid(c32, g_f, c32.with_(layout=0))
    torch.cuda.synchronize()
    assert int(r.workspace[8:12].view(torch.int32).item()) == R * K
    assert dvgo.dvgo_workspace_status(r.workspace) == 0
    ref = oracle.render(oracle_params(p, (RES,) * 3, 12), dens, feat, o, d, mlp=mlp, explicit_t=ts, explicit_dt=dts,
                        grad_rgb=gC, error_bound=BOUND_FP32)
    assert_close(rgb.cpu().numpy(), ref.rgb, RTOL_COLOUR, "rgb")
    assert_close(tf.cpu().numpy(), ref.tfinal, RTOL_COLOUR, "tfinal")
    got = {"rgb": rgb.cpu().numpy(), "g_d": g_d.reshape((RES,) * 3).cpu().numpy(),
           "g_f": g_f.reshape((RES,) * 3 + (12,)).cpu().numpy(), "g_m": g_m.cpu().numpy()}
    _check(got, ref, capsys, f"FP32 {R} x {K}, pe_x {pe_x}, packed {packed}, scale {scale}")
