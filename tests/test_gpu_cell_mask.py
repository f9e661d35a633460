"""The density pass's cell mask (uniform steps, tau_f > 0, batches whose samples outnumber half the cells): a
batch large enough for it renders exactly what the same rays render in batches too small for it -- kept
samples, colours and transmittance bit for bit -- over activation orders, layouts, known free space,
thresholds, steep fields (corners of mixed sign and size), infinite and NaN densities, and a lattice
whose rows are no multiple of 32; rays that terminate and rays without samples included."""
import numpy as np
import pytest
import torch

import synth
from test_gpu_parity import _mlp_flat, cuda

pytestmark = pytest.mark.gpu

dvgo = pytest.importorskip("paper_2111_11215_gb300")

SHAPE, BIG, SMALL = (24, 21, 37), 1024, 8


def _render(p, dd, cd, dens, feat, mlp, o, d, jit, n):
    rend = dvgo.Renderer(p, dd, cd, n)
    out = []
    for s in range(0, o.shape[0], n):
        rgb, tf, _ = rend.forward(dens, feat, mlp, o[s:s + n].contiguous(), d[s:s + n].contiguous(), jit[s:s + n].contiguous())
        kept = rend.workspace[8:12].view(torch.int32).clone()
        out.append((rgb.clone(), tf.clone(), kept))
    torch.cuda.synchronize()
    return (torch.cat([x[0] for x in out]), torch.cat([x[1] for x in out]), int(sum(int(x[2].item()) for x in out)),
            rend.ws_bytes)


@pytest.mark.parametrize("order,packed,fs,tau_f,special", [
    (0, 0, False, 1e-4, False), (0, 1, False, 1e-4, False), (0, 0, True, 1e-3, False), (0, 0, False, 0.3, False),
    (0, 0, False, 1e-4, True), (1, 0, False, 1e-4, False), (2, 1, True, 1e-4, False), (0, 0, False, 1e-12, False),
])
def test_masked_pass_equals_the_plain_one(order, packed, fs, tau_f, special):
    g = np.random.default_rng(11)
    dens = (g.normal(size=SHAPE) * 6.0 + np.where(g.uniform(size=SHAPE) < 0.05, 300.0, -4.0)).astype(np.float32)
    dens[:, :, :9] = -30.0
    if special:
        dens[5, 5, 20], dens[9, 9, 25], dens[3, 12, 30] = np.inf, np.nan, -np.inf
    feat = g.normal(size=SHAPE + (12,)).astype(np.float32)
    mlp = dvgo.mlp_views(cuda(_mlp_flat(synth.mlp_weights(39, 128, 3, 7))))
    o, d, jit, _ = (cuda(a) for a in synth.fine_batch(BIG, 13))
    step = 0.02
    free = None
    if fs:
        free = dvgo.FreeSpace(cuda(g.normal(size=(12, 12, 12)).astype(np.float32) * 4.0),
                              dvgo.GridDesc((12,) * 3, 1), shift_b=-4.0, step=0.05, tau=1e-3)
    p = dvgo.Params(mode=dvgo.DVGO_MODE_FINE, step=step, shift_b=-3.0, tau_f=tau_f, act_order=order, freespace=free,
                    bg=(1.0, 0.5, 0.25))
    dd, cd = dvgo.GridDesc(SHAPE, 1), dvgo.GridDesc(SHAPE, 12)
    D, F = cuda(dens), cuda(feat)
    if packed:
        D, F = dvgo.dvgo_pack_grid(dd, D, dd.with_(layout=1)), dvgo.dvgo_pack_grid(cd, F, cd.with_(layout=1))
        dd, cd = dd.with_(layout=1), cd.with_(layout=1)
    big = _render(p, dd, cd, D, F, mlp, o, d, jit, BIG)
    small = _render(p, dd, cd, D, F, mlp, o, d, jit, SMALL)
    words = SHAPE[0] * SHAPE[1] * 2
    plain = dvgo.dvgo_workspace_size(p.with_(tau_f=0.0), dd, BIG)
    assert big[3] >= plain + 4 * words and small[3] == dvgo.dvgo_workspace_size(p.with_(tau_f=0.0), dd, SMALL)
    assert big[2] == small[2] > 0
    assert torch.equal(big[0].view(torch.int32), small[0].view(torch.int32))
    assert torch.equal(big[1].view(torch.int32), small[1].view(torch.int32))
