"""A workspace sized with tau_f = 0 serves renders with tau_f > 0 (a schedule that turns the skips on later): forward,
backward, labels and touched counts are accepted, with the results of a workspace sized for them; one byte
less than the size at tau_f = 0 is refused."""
import numpy as np
import pytest
import torch

import synth
from test_gpu_parity import _mlp_flat, cuda

pytestmark = pytest.mark.gpu

dvgo = pytest.importorskip("paper_2111_11215_gb300")

RES, R = 24, 1024


@pytest.mark.parametrize("bf16", [False, True])
def test_workspace_sized_without_the_skips_is_accepted(bf16):
    g = np.random.default_rng(61)
    dens = cuda(np.where(g.uniform(size=(RES,) * 3) < 0.7, -30.0, 4.0).astype(np.float32))
    feat = cuda(g.normal(size=(RES,) * 3 + (12,)).astype(np.float32))
    flat = cuda(_mlp_flat(synth.mlp_weights(39, 128, 3, 62)))
    o, d, jit, _ = (cuda(a) for a in synth.fine_batch(R, 63))
    gC = cuda(np.random.default_rng(64).normal(size=(R, 3)).astype(np.float32))
    p0 = dvgo.Params(mode=dvgo.DVGO_MODE_FINE, step=0.04, shift_b=-3.0,
                     mlp_prec=dvgo.DVGO_MLP_BF16 if bf16 else dvgo.DVGO_MLP_FP32)
    p = p0.with_(tau_f=1e-4)
    dd, cd = dvgo.GridDesc((RES,) * 3, 1), dvgo.GridDesc((RES,) * 3, 12)
    assert dvgo.dvgo_workspace_size(p0, dd, R) < dvgo.dvgo_workspace_size(p, dd, R)
    out = []
    for first in (p, p0):
        r = dvgo.Renderer(first, dd, cd, R)
        r.params = p
        views = dvgo.mlp_views(flat)
        rgb, tf, _ = r.forward(dens, feat, views, o, d, jit)
        labels = torch.zeros((R, 64), device="cuda")
        dvgo.dvgo_weight_bins(p, dd, R, 64, r.workspace, labels)
        kept = int(r.workspace[8:12].view(torch.int32).item())
        gd, gf, gm = torch.zeros_like(dens), torch.zeros_like(feat), torch.zeros_like(flat)
        r.backward(dens, feat, views, o, d, jit, None, gC, None, gd, gf, gm)
        torch.cuda.synchronize()
        out.append((rgb.clone(), tf.clone(), labels, kept, gd, gf, gm))
    a, b = out
    assert a[3] == b[3] > 0
    for x, y in zip(a[:3], b[:3]):
        assert torch.equal(x, y)
    for x, y in zip(a[4:], b[4:]):      # (FP32 atomics, and tiles in the order of the kept list)
        torch.testing.assert_close(x, y, rtol=1e-3, atol=1e-4 * float(x.abs().max()))
    small = dvgo.Renderer(p0, dd, cd, R)
    small.workspace = small.workspace[:dvgo.dvgo_workspace_size(p0, dd, R) - 1]
    small.ws_bytes = dvgo.dvgo_workspace_size(p0, dd, R) - 1
    with pytest.raises(dvgo.DVGOError):
        small.forward(dens, feat, views, o, d, jit)
