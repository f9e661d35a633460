"""Weight gradients of the FP32 MLP are sums over samples whose weights span many orders of magnitude.  A tensor core
adds each term cut off at the last bit of the running sum, which loses the same way every time, so a tile's
gradient is kept in several sums that are joined with rounding.  The result must stay as exact as a sum that
rounds: 10 roundings, 10 x 2^-24 in relative L2, against FP64 (FP32 chains over a tile's samples are at 4 to 7 of
them, one cut-off sum for a tile at 13 to 25).  A step of 25 explicit samples a ray as a trained proposal draws them."""
import pytest
import torch

pytestmark = pytest.mark.gpu

dvgo = pytest.importorskip("paper_2111_11215_gb300")


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_weight_gradients_are_not_cut_off(seed):
    import perf.cases as cases
    case = dict(kind="fine", res=64, rays=1000, mlp="fp32", feat="fp32", pe_x=False, skip=False, aux=True, samples=25,
                blob=False)
    state = cases.prepare(case, seed)
    ref = cases.exact(case, seed)["g_mlp"]
    got = cases.run(state)["g_mlp"].double()
    torch.cuda.synchronize()
    a, b = dvgo.mlp_views(got), dvgo.mlp_views(ref)
    for k in ("w1", "b1", "w2"):
        err = float((a[k] - b[k]).norm() / b[k].norm())
        assert err <= 10 * 2 ** -24, (k, err)
