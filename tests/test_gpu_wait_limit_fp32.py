"""Failure detection of the FP32 MLP's tensor-core colour kernels, as for the BF16 ones: one producer arrival is
withheld on a chosen tile (dvgo_params.test_withhold_tile), the consumers' bounded wait for it runs out, the
call returns within a few limits, reports DVGO_ERR_DEVICE, and leaves the context and the tensor memory usable:
the next clean call gives the clean results.  Forward of 39 and 72 inputs, backward of 39; a CTA's first
tile, a later one, and the last."""
import time

import pytest
import torch

from test_gpu_parity import _mlp_flat, cuda
from test_gpu_wait_limit import LIMIT_US, _setup, _step

import synth

pytestmark = pytest.mark.gpu

dvgo = pytest.importorskip("paper_2111_11215_gb300")


@pytest.mark.parametrize("pe_x,bwd", [(0, False), (5, False), (0, True)])
@pytest.mark.parametrize("where", ["first", "later", "last"])
def test_fp32_wait_runs_out_reports_and_leaves_the_context_usable(pe_x, bwd, where):
    p, dd, cd, R, t = _setup()
    p = p.with_(mlp_prec=dvgo.DVGO_MLP_FP32, n_freq_pos=pe_x)
    if pe_x:
        t["flat"] = cuda(_mlp_flat(synth.mlp_weights(72, 128, 3, 702)))
        t["views"] = dvgo.render.mlp_views(t["flat"], 72)
    clean = dvgo.Renderer(p, dd, cd, R)
    ref = _step(clean, t, bwd)
    assert dvgo.dvgo_workspace_status(clean.workspace) == 0
    n_tiles = -(-int(clean.workspace[8:12].view(torch.int32).item()) // 128)
    assert n_tiles > 160            # a CTA with the first tile has later tiles that it must abandon
    tile = {"first": 4, "later": 155, "last": n_tiles}[where]
    faulty = dvgo.Renderer(p, dd, cd, R)
    args = (t["D"], t["F"], t["views"], t["o"], t["d"], t["jit"])
    if bwd:
        faulty.forward(*args)
    torch.cuda.synchronize()
    faulty.params = p.with_(wait_limit_us=LIMIT_US, test_withhold_tile=tile)
    g_m = torch.zeros_like(t["flat"])
    t0 = time.perf_counter()
    if bwd:
        faulty.backward(*args, None, t["gC"], None, torch.zeros_like(t["D"]), torch.zeros_like(t["F"]), g_m)
    else:
        faulty.forward(*args)
    torch.cuda.synchronize()
    dt = time.perf_counter() - t0
    assert dvgo.dvgo_workspace_status(faulty.workspace) == dvgo.binding.DVGO_ERR_DEVICE
    assert dt < 1.0, dt             # a few waits of 20 ms, not the 2 s default
    if bwd:
        assert not torch.equal(g_m, ref["g_m"])
    again = _step(dvgo.Renderer(p, dd, cd, R), t, bwd)
    assert torch.equal(again["rgb"], ref["rgb"])
    for k in ("g_d", "g_f", "g_m") if bwd else ():
        torch.testing.assert_close(again[k], ref[k], rtol=1e-4, atol=1e-4 * float(ref[k].abs().max()))
