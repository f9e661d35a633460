"""Feature gradients of samples on the rim of the box, against the FP64 oracle: explicit samples at the entry
point, a little outside or inside it by the rounding of t, then a few more in the same and the next cell, and
the same at the exit.  The offset of such a sample inside its cell is a little below 0 or above 1, and
consecutive rows of a tile share the cell or corners of it.  64 rays x 8 samples and a ragged last tile; both
layouts and both MLP paths; BF16 inputs where the path rounds them.  Tolerances as everywhere: the oracle's
running error bound of the path."""
import numpy as np
import pytest
import torch

import oracle
import synth
from helpers import BOUND_BF16_OPERANDS, BOUND_FP32, mlp_flat, oracle_params
from test_gpu_bf16_tiles import _bf16, _check
from test_gpu_fine_edges import RES, _bf16_operands, _hitting_rays, _params
from test_gpu_parity import _fine_inputs

pytestmark = pytest.mark.gpu

dvgo = pytest.importorskip("paper_2111_11215_gb300")

R, K = 77, 8


def _rim_samples():
    voxel = 2.0 / (RES - 1)
    o, d, t0, t1 = _hitting_rays(2 * R, 841)
    long = np.nonzero(t1 - t0 > 3 * voxel)[0][:R]
    assert len(long) == R
    o, d, t0, t1 = o[long], d[long], t0[long], t1[long]
    off = np.array([0.0, 0.15, 0.3, 0.9]) * voxel
    t = np.concatenate([t0[:, None] + off, t1[:, None] - off[::-1]], axis=1)
    ts = np.sort(t, axis=1).astype(np.float32)
    dts = np.full(ts.shape, 0.25 * voxel, np.float32)
    e = np.asarray(d, np.float64) / np.linalg.norm(d, axis=1, keepdims=True)
    u = (np.asarray(o, np.float64)[:, None] + ts[..., None].astype(np.float64) * e[:, None] + 1.0) / voxel
    return o, d, ts, dts, u


@pytest.mark.parametrize("packed", [0, 1])
@pytest.mark.parametrize("bf16", [False, True])
def test_rim_samples_match_oracle(bf16, packed, capsys):
    dens, feat, mlp, _, _, _, _ = _fine_inputs(RES, 8, seed=840)
    if bf16:
        feat = _bf16(feat)
    o, d, ts, dts, u = _rim_samples()
    assert (u < 0).any(axis=2).sum() > R // 4 and (u > RES - 1).any(axis=2).sum() > R // 4
    p = _params(dvgo.DVGO_MLP_BF16 if bf16 else dvgo.DVGO_MLP_FP32)
    gC = np.random.default_rng(842).normal(scale=1e-2, size=(R, 3))
    dd = dvgo.GridDesc((RES,) * 3, 1)
    cd = dvgo.GridDesc((RES,) * 3, 12)
    cu = lambda a, t=torch.float32: torch.as_tensor(np.ascontiguousarray(a)).to(device="cuda", dtype=t)  # noqa: E731
    D, F, flat = cu(dens), cu(feat), cu(mlp_flat(mlp))
    if packed:
        D, F = dvgo.dvgo_pack_grid(dd, D, dd.with_(layout=1)), dvgo.dvgo_pack_grid(cd, F, cd.with_(layout=1))
        dd, cd = dd.with_(layout=1), cd.with_(layout=1)
    views = dvgo.render.mlp_views(flat, 39)
    r = dvgo.Renderer(p, dd, cd, R, samples_per_ray=K)
    samples = (cu(ts), cu(dts))
    rgb, _, _ = r.forward(D, F, views, cu(o), cu(d), None, samples)
    g_d, g_f, g_m = torch.zeros_like(D), torch.zeros_like(F), torch.zeros_like(flat)
    r.backward(D, F, views, cu(o), cu(d), None, samples, cu(gC), None, g_d, g_f, g_m)
    if packed:
        g_d, g_f = dvgo.dvgo_pack_grid(dd, g_d, dd.with_(layout=0)), dvgo.dvgo_pack_grid(cd, g_f, cd.with_(layout=0))
    torch.cuda.synchronize()
    assert int(r.workspace[8:12].view(torch.int32).item()) == R * K
    ref = oracle.render(oracle_params(p, (RES,) * 3, 12, bf16_operands=bf16), dens, feat, o, d,
                        mlp=_bf16_operands(mlp) if bf16 else mlp, explicit_t=ts, explicit_dt=dts, grad_rgb=gC,
                        error_bound=BOUND_BF16_OPERANDS if bf16 else BOUND_FP32)
    got = {"rgb": rgb.cpu().numpy(), "g_d": g_d.reshape((RES,) * 3).cpu().numpy(),
           "g_f": g_f.reshape((RES,) * 3 + (12,)).cpu().numpy(), "g_m": g_m.cpu().numpy()}
    _check(got, ref, capsys, f"rim, {'BF16' if bf16 else 'FP32'}, packed {packed}")
