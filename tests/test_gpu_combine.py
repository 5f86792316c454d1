"""The Weight Sum at every number of slots in flight (1, 2, 4, 8 and groups of
them), with few tokens (a block per 1024 columns) and many (a block walks a row),
dropped pairs among them."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_12875_gb300 as gb
from gpu_helpers import act_np, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("act", ["f32", "bf16"])
@pytest.mark.parametrize("T", [3, 2600])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 8, 9, 12])
def test_slots_and_blocks(T, k, act):
    rng = np.random.default_rng(k)
    H, dt = 1280, torch.float32 if act == "f32" else torch.bfloat16
    cfg = gb.make_config(T, H, 128, 16, k, act=act, w="bf16" if act == "bf16" else "f32")
    y = torch.from_numpy(rng.standard_normal((T * k, H)).astype(np.float32)).cuda().to(dt)
    ysh = torch.from_numpy(rng.standard_normal((T, H)).astype(np.float32)).cuda().to(dt)
    w = rng.random((T, k)).astype(np.float32)
    pp = rng.permutation(T * k).astype(np.int32).reshape(T, k)
    dropped = rng.random((T, k)) < 0.1
    pos = torch.from_numpy(np.where(dropped, -1, pp).astype(np.int32)).cuda()
    out = torch.empty((T, H), dtype=dt, device="cuda")
    for shared in (None, ysh):
        gb.moe_combine(cfg, y, torch.from_numpy(w).cuda(), pos, shared, out)
        torch.cuda.synchronize()
        ref = oracle.combine(act_np(y), np.where(dropped, 0.0, w).astype(np.float64), pp,
                             None if shared is None else act_np(shared))
        # fp32 sums of up to 13 terms; one rounding to bf16 (2^-9 of a value) on top
        assert rel_err(act_np(out), ref) <= (1e-6 if act == "f32" else 4e-3)
