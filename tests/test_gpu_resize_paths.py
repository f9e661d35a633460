"""The resize kernel's splits against the FP64 oracle: chunks of z (more destination points than one
holds, and a span limited by the channel count), a destination coarser than half the source (two
source points per destination point), more channels than one block takes, single rows, and values
that are infinite or NaN.  Tolerance: the FP32 rounding of the result, 2^-24 relative, taken twice;
atol covers values that cancel (the sum is kept to ~2^-46 of its largest term, |terms| <= ~5)."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_parity import cuda

pytestmark = pytest.mark.gpu

dvgo = pytest.importorskip("paper_2111_11215_gb300")


@pytest.mark.parametrize("C,src,dst,layouts", [
    (1, (3, 4, 300), (2, 3, 611), (0, 0)),        # three chunks along z
    (12, (4, 3, 230), (3, 5, 290), (0, 1)),       # chunks shortened by the shared-memory row
    (12, (3, 5, 257), (4, 2, 40), (0, 0)),        # 6.6 source points per destination point
    (3, (2, 2, 2), (2, 2, 2), (0, 0)),            # the smallest lattice
    (12, (5, 4, 64), (3, 3, 33), (1, 0)),         # just above and below two points per point
    (12, (5, 4, 64), (3, 3, 32), (1, 1)),
    (70, (3, 3, 20), (4, 3, 27), (0, 0)),         # two channel chunks
])
def test_resize_splits_match_oracle(C, src, dst, layouts):
    g = np.random.default_rng(3 + C)
    a = g.normal(size=tuple(src) + ((C,) if C > 1 else ())).astype(np.float32)
    sd, dd = dvgo.GridDesc(src, C), dvgo.GridDesc(dst, C)
    x = cuda(a).reshape(-1)
    if layouts[0]:
        x = dvgo.dvgo_pack_grid(sd, x, sd.with_(layout=1))
    out = dvgo.dvgo_resize_grid(sd.with_(layout=layouts[0]), x, dd.with_(layout=layouts[1]))
    if layouts[1]:
        out = dvgo.dvgo_pack_grid(dd.with_(layout=1), out, dd)
    got = out.reshape(tuple(dst) + ((C,) if C > 1 else ())).cpu().numpy()
    np.testing.assert_allclose(got, oracle.resize_grid(a, dst), rtol=2 ** -23, atol=1e-12)


def test_resize_keeps_infinities_and_nan():
    a = np.ones((4, 4, 4), dtype=np.float32)
    a[1, 1, 1], a[3, 3, 3] = np.inf, np.nan
    got = dvgo.dvgo_resize_grid(dvgo.GridDesc((4, 4, 4), 1), cuda(a).reshape(-1),
                                dvgo.GridDesc((6, 6, 6), 1)).reshape(6, 6, 6).cpu().numpy()
    u = np.arange(6) * 3 / 5
    near = (np.abs(u - 1) < 0.99).astype(int)            # a corner of weight > 0.01 on an axis
    inf = near[:, None, None] * near[None, :, None] * near[None, None, :] == 1
    assert np.isinf(got[inf]).all() and (got[inf] > 0).all()
    assert np.isnan(got[5, 5, 5]) and got[0, 0, 5] == 1.0
