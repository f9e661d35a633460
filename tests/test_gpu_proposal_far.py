"""The FP32 proposal network far from the origin (a scene in projected map coordinates): positions and argument
reductions keep FP64, so the probabilities match an FP64 evaluation to 1e-6 in relative L2 (at 1e10 an FP64 position
is off by 32 x 1e10 x 2^-53 = 4e-5 in the highest encoded argument, and a hundredth of that reaches the
probabilities; positions of 48 bits are off by 32 times as much).  The same near the origin as a control."""
import numpy as np
import pytest
import torch

from test_gpu_parity import cuda
from test_gpu_proposal import NB, NFQ, PW, _proposal_weights

pytestmark = pytest.mark.gpu

dvgo = pytest.importorskip("paper_2111_11215_gb300")

R = 75


def _reference(o, d, lo3, hi3, w):
    o, d = o.astype(np.float64), d.astype(np.float64)
    dn = d / np.sqrt((d[:, :1] * d[:, :1] + d[:, 1:2] * d[:, 1:2]) + d[:, 2:] * d[:, 2:])
    t1, t2 = (lo3 - o) / dn, (hi3 - o) / dn
    lo, hi = np.maximum(np.minimum(t1, t2).max(1), 0.0), np.maximum(t1, t2).min(1)
    assert (hi > lo).all()
    tb = lo[:, None] + ((np.arange(NB) + 0.5) * (hi - lo)[:, None]) / NB
    x = o[:, None, :] + tb[..., None] * dn[:, None, :]
    a = x[..., None] * 2.0 ** np.arange(NFQ)
    h = np.concatenate([x, np.sin(a).reshape(R, NB, -1), np.cos(a).reshape(R, NB, -1)], -1)
    for i in range(3):
        h = np.maximum(h @ w[f"w{i}"].astype(np.float64) + w[f"b{i}"], 0.0)
    z = (h @ w["w3"].astype(np.float64).reshape(PW, 1))[..., 0] + w["b3"]
    e = np.exp(z - z.max(1, keepdims=True))
    return e / e.sum(1, keepdims=True)


@pytest.mark.parametrize("centre,half", [((0.0, 0.0, 0.0), 1.0), ((1e10, -9e9, 5e9), 65536.0)])
def test_far_positions_keep_fp64(centre, half):
    g = np.random.default_rng(91)
    c = np.array(centre).astype(np.float32).astype(np.float64)
    v = g.normal(size=(R, 3))
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    o = (c + 4.0 * half * v).astype(np.float32)
    target = c + half * g.uniform(-0.5, 0.5, size=(R, 3))
    d = (target - o).astype(np.float32)
    lo3, hi3 = (c - half).astype(np.float32), (c + half).astype(np.float32)
    w = _proposal_weights(92)
    # inputs of size 1e10 would drown the encoded ones: the raw coordinates stay out of the first layer
    if half > 1.0:
        w["w0"][:3] = 0.0
    dd = dvgo.GridDesc((16,) * 3, 1, xyz_min=tuple(lo3.tolist()), xyz_max=tuple(hi3.tolist()))
    p = dvgo.Params(mode=dvgo.DVGO_MODE_FINE, step=0.05 * half)
    probs = torch.empty((R, NB), device="cuda")
    dvgo.dvgo_proposal_fwd(p, dd, NB, NFQ, PW, {k: cuda(x) for k, x in w.items()}, cuda(o), cuda(d), None, probs, None)
    torch.cuda.synchronize()
    ref = _reference(o, d, lo3.astype(np.float64), hi3.astype(np.float64), w)
    err = np.linalg.norm(probs.double().cpu().numpy() - ref) / np.linalg.norm(ref)
    assert err <= 1e-6, err
