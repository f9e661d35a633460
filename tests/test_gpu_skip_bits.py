"""What the skips leave out changes no bit of what stays: a batch rendered with a tau_f so small that it removes only
samples whose optical depth is lost in every sum (alpha < 1e-30 against sums above 1e-3) has the colours, the
transmittance, the loss gradient and the proposal's labels of the same batch rendered with every sample,
bit for bit -- sums over a ray are associated by the sample's place along it, not by its place among the kept
ones.  BF16 roundings of dL/do then agree too: the feature gradients differ by the order of FP32 sums
alone (at most 200 terms a corner: 200 x 2^-24 of their magnitude; one flipped BF16 rounding of a leading
term is 2^-9 of it)."""
import numpy as np
import pytest
import torch

import synth
from test_gpu_parity import _mlp_flat, cuda

pytestmark = pytest.mark.gpu

dvgo = pytest.importorskip("paper_2111_11215_gb300")

RES, R, K = 40, 700, 90


def _inputs():
    g = np.random.default_rng(51)
    dens = np.where(g.uniform(size=(RES,) * 3) < 0.12, -400.0, g.normal(size=(RES,) * 3) * 2.0 + 2.0)
    feat = g.normal(size=(RES,) * 3 + (12,))
    o, d, jit, tgt = synth.fine_batch(R, 52)
    return [cuda(np.asarray(a, np.float32)) for a in (dens, feat, o, d, jit, tgt)]


@pytest.mark.parametrize("prec,explicit", [(0, False), (1, False), (1, True)])
def test_skips_change_no_bit_of_the_rest(prec, explicit):
    dens, feat, o, d, jit, tgt = _inputs()
    flat = cuda(_mlp_flat(synth.mlp_weights(39, 128, 3, 53)))
    samples = None
    if explicit:
        g = np.random.default_rng(54)
        t = np.sort(g.uniform(2.4, 5.6, size=(R, K)), axis=1)
        samples = (cuda(t.astype(np.float32)), cuda(np.full((R, K), 0.03, np.float32)))
    dd, cd = dvgo.GridDesc((RES,) * 3, 1), dvgo.GridDesc((RES,) * 3, 12)
    out = []
    for tau_f in (0.0, 1e-30):
        p = dvgo.Params(mode=dvgo.DVGO_MODE_FINE, step=0.5 * 2.0 / RES, shift_b=-4.0, tau_f=tau_f, bg=(1.0, 0.5, 0.25),
                        mlp_prec=dvgo.DVGO_MLP_BF16 if prec else dvgo.DVGO_MLP_FP32, w_pt_rgb=0.01)
        r = dvgo.Renderer(p, dd, cd, R, samples_per_ray=K if explicit else None)
        views = dvgo.mlp_views(flat)
        dloss = torch.empty((R, 3), device="cuda")
        rgb, tf, _ = r.forward(dens, feat, views, o, d, jit, samples, tgt, dloss=dloss)
        kept = int(r.workspace[8:12].view(torch.int32).item())
        labels = torch.zeros((R, 64), device="cuda")
        if not explicit:
            dvgo.dvgo_weight_bins(p, dd, R, 64, r.workspace, labels)
        gd, gf, gm = torch.zeros_like(dens), torch.zeros_like(feat), torch.zeros_like(flat)
        r.backward(dens, feat, views, o, d, jit, samples, dloss, None, gd, gf, gm)
        torch.cuda.synchronize()
        out.append((kept, [x.clone() for x in (rgb, tf, dloss, labels)], gf))
    (all_kept, a, ga), (some, b, gb) = out
    assert 0.2 * all_kept < some < 0.8 * all_kept, (some, all_kept)
    for name, x, y in zip(("rgb", "tfinal", "dloss", "labels"), a, b):
        big = x.abs() > 1e-20          # (a bin of removed samples alone holds up to 1e-30)
        assert torch.equal(x[big].view(torch.int32), y[big].view(torch.int32)), (name, int((x != y).sum()))
    assert float((ga - gb).abs().max() / ga.abs().max()) <= 200 * 2 ** -24
