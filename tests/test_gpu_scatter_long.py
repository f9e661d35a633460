"""Feature gradients on a packed lattice of more than 1024 points along x (the layout takes up to 2048), against
the FP64 oracle: explicit samples along rays nearly parallel to x, below, across and above i = 1024, several
to a cell, a ragged last tile; both MLP paths.  Tolerances as everywhere: the oracle's running error bound of
the path."""
import numpy as np
import pytest
import torch

import oracle
import synth
from helpers import BOUND_BF16_OPERANDS, BOUND_FP32, mlp_flat, oracle_params
from test_gpu_bf16_tiles import _bf16, _check
from test_gpu_fine_edges import _bf16_operands, _params

pytestmark = pytest.mark.gpu

dvgo = pytest.importorskip("paper_2111_11215_gb300")

SHAPE, R, K = (1100, 6, 7), 45, 16


@pytest.mark.parametrize("bf16", [False, True])
def test_long_packed_lattice_matches_oracle(bf16, capsys):
    g = np.random.default_rng(861)
    dens = g.normal(size=SHAPE).astype(np.float32)
    feat = g.normal(size=SHAPE + (12,)).astype(np.float32)
    mlp = synth.mlp_weights(39, 128, 3, 862)
    if bf16:
        feat = _bf16(feat)
    o = np.stack([np.full(R, -2.0), g.uniform(-0.8, 0.8, R), g.uniform(-0.8, 0.8, R)], 1).astype(np.float32)
    d = np.stack([np.ones(R), g.uniform(-0.03, 0.03, R), g.uniform(-0.03, 0.03, R)], 1).astype(np.float32)
    u0 = np.array([1020.3, 300.1, 1060.7])[np.arange(R) % 3] + g.uniform(0, 1, R)      # first sample's lattice x
    x = (u0[:, None] + 0.45 * np.arange(K)) * 2.0 / (SHAPE[0] - 1) - 1.0
    ts = ((x - o[:, :1]) * np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32)
    dts = np.full((R, K), 1e-3, np.float32)
    p = _params(dvgo.DVGO_MLP_BF16 if bf16 else dvgo.DVGO_MLP_FP32)
    gC = g.normal(scale=1e-2, size=(R, 3))
    dd, cd = dvgo.GridDesc(SHAPE, 1), dvgo.GridDesc(SHAPE, 12)
    cu = lambda a: torch.as_tensor(np.ascontiguousarray(a)).to(device="cuda", dtype=torch.float32)  # noqa: E731
    D, F, flat = cu(dens), cu(feat), cu(mlp_flat(mlp))
    D, F = dvgo.dvgo_pack_grid(dd, D, dd.with_(layout=1)), dvgo.dvgo_pack_grid(cd, F, cd.with_(layout=1))
    dd, cd = dd.with_(layout=1), cd.with_(layout=1)
    views = dvgo.render.mlp_views(flat, 39)
    r = dvgo.Renderer(p, dd, cd, R, samples_per_ray=K)
    samples = (cu(ts), cu(dts))
    rgb, _, _ = r.forward(D, F, views, cu(o), cu(d), None, samples)
    g_d, g_f, g_m = torch.zeros_like(D), torch.zeros_like(F), torch.zeros_like(flat)
    r.backward(D, F, views, cu(o), cu(d), None, samples, cu(gC), None, g_d, g_f, g_m)
    g_d, g_f = dvgo.dvgo_pack_grid(dd, g_d, dd.with_(layout=0)), dvgo.dvgo_pack_grid(cd, g_f, cd.with_(layout=0))
    torch.cuda.synchronize()
    assert int(r.workspace[8:12].view(torch.int32).item()) == R * K
    ref = oracle.render(oracle_params(p, SHAPE, 12, bf16_operands=bf16), dens, feat, o, d,
                        mlp=_bf16_operands(mlp) if bf16 else mlp, explicit_t=ts, explicit_dt=dts, grad_rgb=gC,
                        error_bound=BOUND_BF16_OPERANDS if bf16 else BOUND_FP32)
    assert np.abs(ref.grads["cgrid"][1026:]).max() > 0 and np.abs(ref.grads["cgrid"][:1024]).max() > 0
    got = {"rgb": rgb.cpu().numpy(), "g_d": g_d.reshape(SHAPE).cpu().numpy(),
           "g_f": g_f.reshape(SHAPE + (12,)).cpu().numpy(), "g_m": g_m.cpu().numpy()}
    _check(got, ref, capsys, f"long packed lattice, {'BF16' if bf16 else 'FP32'}")
