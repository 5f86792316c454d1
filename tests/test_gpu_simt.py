"""The CUDA-core GEMM against the oracle at the edges of its row tiles for every
weight format: 32 rows x 64 weight rows for small problems, then 64 x 128 (1001
tokens), 64 x 128 with a down GEMM of 64 x 64 (700) and 32 x 128 (600)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_12875_gb300 as gb
import synth
from gpu_helpers import act_np, assert_close, config, to_device, tol_for, wbundle, workspace

pytestmark = pytest.mark.gpu

BASE = synth.WORKLOADS[1]


@pytest.mark.parametrize("act,wq", [("f32", "f32"), ("f32", "bf16"), ("f32", "fp8_b128"), ("f32", "int4_g128"),
                                    ("f32", "mxfp4"), ("bf16", "bf16"), ("bf16", "fp8_b128")])
@pytest.mark.parametrize("T,E,k,H,I", [(1, 2, 1, 256, 128), (32, 1, 1, 256, 128), (40, 1, 1, 512, 384),
                                       (41, 1, 1, 512, 128), (65, 1, 1, 256, 256), (200, 3, 2, 768, 128),
                                       (1001, 16, 4, 1024, 768), (700, 16, 4, 1024, 768), (600, 64, 2, 2048, 1024)])
def test_row_tiles(T, E, k, H, I, act, wq):
    wl = BASE.replace(T=T, E=E, top_k=k, H=H, I=I, act=act, wq=wq, seed=T + E)
    inp = synth.make_inputs(wl)
    dev = to_device(wl, inp)
    cfg = config(wl, "simt")
    ws = workspace(cfg)
    out = torch.empty((wl.T, wl.H), dtype=dev["x"].dtype, device="cuda")
    gb.moe_forward(cfg, dev["x"], dev["w_router"], None, None, wbundle(dev["experts"]), None, out, ws)
    torch.cuda.synchronize()
    # fp32 sums of the formats' exact decodings: 1e-5 for fp32 activations
    assert_close(act_np(out), oracle.forward(wl, inp)["out"], 1e-5 if act == "f32" else tol_for(wl))
