"""The streaming route with fp32 weights against the oracle where it takes one
CTA per SM (a grid of few CTAs; activation rows that two CTAs' L1 share could not
spare) and two, with one pass of 8 rows per expert and several."""
import pytest
import torch

import oracle
import paper_2607_12875_gb300 as gb
import synth
from gpu_helpers import act_np, assert_close, config, to_device, wbundle, workspace

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,E,k,H,I", [(3, 1, 1, 512, 256), (16, 1, 1, 3584, 128), (12, 4, 2, 3584, 3328),
                                       (40, 16, 2, 1024, 256), (77, 16, 2, 256, 512)])
def test_fp32_ctas_per_sm(T, E, k, H, I):
    wl = synth.WORKLOADS[1].replace(T=T, E=E, top_k=k, H=H, I=I, seed=T)
    inp = synth.make_inputs(wl)
    dev = to_device(wl, inp)
    cfg = config(wl, "stream")
    ws = workspace(cfg)
    out = torch.empty((T, H), dtype=torch.float32, device="cuda")
    gb.moe_forward(cfg, dev["x"], dev["w_router"], None, None, wbundle(dev["experts"]), None, out, ws)
    torch.cuda.synchronize()
    assert_close(act_np(out), oracle.forward(wl, inp)["out"], 1e-5)
