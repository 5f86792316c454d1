"""The feature-major GEMM (quantised weights as the M operand of tcgen05.mma),
which AUTO takes for few rows per expert, against the oracle at the edges of
its row tiles, and with activations that are not finite."""
import numpy as np
import pytest
import torch

import oracle
import paper_2607_12875_gb300 as gb
import synth
from gpu_helpers import act_np, assert_close, config, to_device, tol_for, wbundle, workspace

pytestmark = pytest.mark.gpu

BASE = synth.WORKLOADS[1].replace(act="bf16")


# the feature-major GEMM's last row per expert, what runs beyond it, and the rows
# (less one) times H * I / (H + I) up to which the weights are streamed instead
LIMITS = {"bf16": (40, "tc", 12000), "fp8_b128": (52, "tc_fp8", 5000), "int4_g128": (40, "tc", 4800),
          "mxfp4": (64, "tc", 1600)}


def few_rows(wq, H, I):
    return 1 + int(LIMITS[wq][2] * (1 / H + 1 / I))


def kernel_of(wl):
    most, beyond, _ = LIMITS[wl.wq]
    if wl.wq == "fp8_b128" and wl.H < 1024:  # few k blocks
        most = 40 if wl.H >= 512 else 28
    joins = wl.has_shared and wl.I_shared == wl.I and wl.wq != "bf16" and wl.P > 1
    few = wl.P <= min(few_rows(wl.wq, wl.H, wl.I), 16 * wl.E) and not joins
    if few or (wl.wq == "bf16" and wl.P < wl.E):
        return "stream"
    return "fm" if wl.P <= most * wl.E else beyond


def tol(wl, kernel="fm"):
    """1e-2 for the feature-major GEMM, whose activation codes keep bf16's
    precision and whose weights are exact: h and y rounded to bf16 give up to 5e-3
    of a row's largest value (0.004 to 0.005 measured). Without the second codes
    these rows are 0.04 to 0.06 off. Other kernels: tol_for."""
    return 1e-2 if kernel == "fm" else tol_for(wl)


def forward(wl, dev, kernel="fm"):
    cfg = config(wl)
    assert gb.ffn_kernel(cfg) == kernel
    ws = workspace(cfg)
    out = torch.empty((wl.T, wl.H), dtype=torch.bfloat16, device="cuda")
    gb.moe_forward(cfg, dev["x"], dev["w_router"], dev["logit_bias"], dev["select_bias"], wbundle(dev["experts"]),
                   wbundle(dev["shared"]), out, ws)
    torch.cuda.synchronize()
    assert gb.moe_device_status(ws) == gb.OK
    return out


@pytest.mark.parametrize("wq", list(LIMITS))
def test_which_kernels_run(wq):
    """The route is AUTO's choice by rows per expert; the kernels reported are
    those launched, on both sides of each limit, for forced routes and for a
    shared expert in the routed launches or by itself."""
    most, other, _ = LIMITS[wq]
    cfg = lambda T, **kw: gb.make_config(T, 4096, 4096, 4, 1, act="bf16", w=wq, **kw)
    assert gb.ffn_kernel(cfg(4 * most)) == "fm"
    assert gb.ffn_kernel(cfg(4 * most + 1)) == other == gb.ffn_route(cfg(4 * most + 1))
    if wq == "fp8_b128":
        for H, last in ((256, 28), (512, 40), (768, 40), (1024, 52)):
            narrow = lambda rows: gb.make_config(4 * rows, H, 4096, 4, 1, act="bf16", w=wq)
            assert gb.ffn_kernel(narrow(last)) == "fm" and gb.ffn_kernel(narrow(last + 1)) == "tc_fp8"
    assert gb.ffn_kernel(cfg(40, ffn_route="simt")) == "simt"
    assert gb.ffn_kernel(cfg(40, ffn_route="tc")) == "tc"
    if wq == "bf16":
        deep = lambda T: gb.make_config(T, 4096, 4096, 16, 1, act="bf16", w=wq)
        assert gb.ffn_kernel(deep(15)) == "stream" and gb.ffn_kernel(deep(16)) == "fm"
        assert gb.ffn_route(deep(16)) == "stream" and gb.ffn_route(deep(257)) == "tc"
    else:
        assert gb.ffn_route(cfg(40)) == ("tc_fp8" if wq == "fp8_b128" else "tc")
    same = dict(has_shared=True, I_shared=4096)
    assert gb.ffn_kernel(cfg(40, **same), shared=True) == ("fm" if wq == "bf16" else "joined")
    assert gb.ffn_kernel(cfg(40, has_shared=True, I_shared=2048), shared=True) == "fm"
    assert gb.ffn_kernel(cfg(2, **same), shared=True) == ("stream" if wq == "bf16" else "joined")
    assert gb.ffn_kernel(cfg(2, has_shared=True, I_shared=2048), shared=True) == "stream"
    assert gb.ffn_kernel(cfg(40, ffn_route="tc", **same), shared=True) == "tc"
    wide = gb.make_config(513, 4096, 4096, 64, 1, act="bf16", w=wq, **same)  # more tokens than join
    assert gb.ffn_kernel(wide) == "fm" and gb.ffn_kernel(wide, shared=True) == gb.ffn_route(wide, shared=True)


# rows per expert: 1, groups of 8 and one more, whole 16-row tiles, the last
# size with the shortest tiles (4 rows per expert on average), 16 and 17 (the next
# tile height) and the first without,
# the last before the row-major GEMM takes over; one k block and ragged rings
# (few rows of small matrices are streamed: the last six are large enough)
@pytest.mark.parametrize("wq", ["bf16", "fp8_b128", "int4_g128", "mxfp4"])
@pytest.mark.parametrize("T,E,k,H,I", [(1, 8, 2, 256, 128), (8, 4, 1, 512, 128), (9, 1, 1, 256, 256),
                                       (4, 1, 1, 768, 384), (32, 16, 2, 1024, 128), (33, 16, 2, 256, 640),
                                       (40, 1, 1, 512, 256), (63, 4, 2, 1280, 256),
                                       (16, 1, 1, 512, 128), (17, 1, 1, 512, 128), (52, 1, 1, 256, 384), (53, 1, 1, 256, 128),
                                       (8, 64, 2, 1024, 512), (8, 2, 1, 4096, 4096), (40, 10, 1, 1024, 512),
                                       (9, 1, 1, 4096, 2560), (16, 1, 1, 2048, 1536), (32, 16, 2, 1024, 256)])
def test_row_tiles(T, E, k, H, I, wq):
    wl = BASE.replace(T=T, E=E, top_k=k, H=H, I=I, wq=wq, seed=T + 7 * E)
    inp = synth.make_inputs(wl)
    out = forward(wl, to_device(wl, inp), kernel_of(wl))
    assert_close(act_np(out), oracle.forward(wl, inp)["out"], tol(wl, kernel_of(wl)))


@pytest.mark.parametrize("E,k", [(1, 1), (8, 2)])
@pytest.mark.parametrize("wq", list(LIMITS))
def test_few_rows_are_streamed(wq, E, k):
    """The last size whose weights are streamed and the first that takes the
    feature-major GEMM, against the oracle and against each other's rows."""
    wl = BASE.replace(E=E, top_k=k, H=2048, I=1024, wq=wq, seed=E)
    last = min(few_rows(wq, wl.H, wl.I), 16 * E) // k
    for T, kernel in ((last, "stream"), (last + 1, "fm")):
        w = wl.replace(T=T)
        assert kernel_of(w) == kernel
        inp = synth.make_inputs(w)
        assert_close(act_np(forward(w, to_device(w, inp), kernel)), oracle.forward(w, inp)["out"], tol(w, kernel))


@pytest.mark.parametrize("wq", ["bf16", "fp8_b128", "int4_g128", "mxfp4"])
@pytest.mark.parametrize("T", [16, 17, 32, 33, 80, 81, 200])
def test_all_rows_on_one_expert(T, wq):
    """A hot expert's rows fill whole row tiles and spill into the next."""
    wl = BASE.replace(T=T, E=16, top_k=2, H=2048, I=512, wq=wq, seed=T)
    inp = synth.make_inputs(wl)
    bias = np.zeros(wl.E, np.float32)
    bias[3] = 1000.0
    inp["logit_bias"] = bias
    ref = oracle.forward(wl, inp)
    assert ref["counts"][3] == T
    assert_close(act_np(forward(wl, to_device(wl, inp))), ref["out"], tol(wl))


@pytest.fixture(scope="module", params=list(LIMITS))
def many_items(request):
    """A layer whose two GEMMs have more items than a GB300 has SMs at every tile
    height, so that CTAs take two items and more: its inputs and the oracle's
    outputs, which tokens share only through the weights."""
    wl = BASE.replace(T=384, E=24, top_k=2, H=2048, I=2048, wq=request.param, seed=21)
    inp = synth.make_inputs(wl)
    return wl, to_device(wl, inp), oracle.forward(wl, inp)["out"]


@pytest.mark.parametrize("T", [48, 192, 384])
def test_more_items_than_sms(many_items, T):
    """16-, 32- and 80-row tiles (bf16: 16 and 64), the same bits from call to call."""
    wl, dev, ref = many_items
    wl = wl.replace(T=T)
    dev = dict(dev, x=dev["x"][:T])
    out = forward(wl, dev)
    assert_close(act_np(out), ref[:T], tol(wl))
    assert torch.equal(out.view(torch.int16), forward(wl, dev).view(torch.int16))


@pytest.mark.parametrize("wq", ["bf16", "fp8_b128", "int4_g128", "mxfp4"])
def test_not_finite_rows_stay_in_their_token(wq):
    """An infinity or NaN in one token's activations leaves every other token's
    output bit for bit as it was; its own output is not finite. Values whose
    squares or quotients would leave fp32's range are scaled exactly."""
    wl = BASE.replace(T=24, E=8, top_k=2, H=1024, I=512, wq=wq, seed=5)
    inp = synth.make_inputs(wl)
    dev = to_device(wl, inp)
    # the experts are fixed by a bias, so that the routing does not depend on the rows changed below
    dev["logit_bias"] = torch.arange(wl.E, device="cuda", dtype=torch.float32) * 1e6
    a = forward(wl, dev)
    for t, v in ((3, float("inf")), (4, float("nan")), (5, float("-inf"))):
        dev["x"][t, 130] = v
    dev["x"][6] = 0
    dev["x"][7] *= 1e-38
    b = forward(wl, dev)
    same = [t for t in range(wl.T) if t not in (3, 4, 5, 6, 7)]
    assert torch.equal(a[same].view(torch.int16), b[same].view(torch.int16))
    assert all(not torch.isfinite(b[t].float()).all() for t in (3, 4, 5))
    assert torch.isfinite(b[6:8].float()).all() and float(b[6].float().abs().max()) == 0.0


CODED = ["fp8_b128", "int4_g128", "mxfp4"]


def one_hot(wq, rows, K):
    """[1, rows, K] weights in the format wq, row n being 1.0 at k = n where there is such a k."""
    n = np.arange(min(rows, K))
    if wq == "fp8_b128":
        w = np.zeros((1, rows, K), np.uint8)
        w[0, n, n] = 0x38
        return w, np.ones((1, rows // 128, K // 128), np.float32)
    w = np.zeros((1, rows, K // 2), np.uint8)
    w[0, n, n // 2] = (2 if wq == "mxfp4" else 1) << (4 * (n % 2)).astype(np.uint8)
    if wq == "mxfp4":
        return w, np.full((1, rows, K // 32), 127, np.uint8)
    return w, np.full((1, rows, K // 128), 0x3F80, np.uint16)


# all rows on one of eight experts: 16-, 32- and 80-row tiles; fp8: the row-major GEMM's 128-row tiles, a pass
# for each code, and a last one of 64 rows with both codes stacked
@pytest.mark.parametrize("spread", [9, 24])
@pytest.mark.parametrize("wq,T", [(wq, T) for wq in CODED for T in (32, 128, 320)] + [("fp8_b128", 448)])
def test_activation_codes_keep_every_value(wq, T, spread):
    """Every element of x, and every element of h, on its own way through the
    two-code activations: gate rows pick a constant, up and down rows one element
    each, so out[t, n] = bf16(silu(g) * x[t, n]). All values are positive and
    most of them large, so that a block's sum is 2^15 times its smallest value.
    Within 2^9 of each other the two codes hold them exactly, and each comes out
    within bf16 rounding; over 2^24 there is also (for x and for h) half of the
    second code's lowest bit, 2^-22 of the block's largest value (row-major GEMM:
    2^-17, the largest being at least 224 and the bit 2^-9)."""
    E, H, I = 8, 512, 256
    rng = np.random.default_rng(T)
    x = rng.uniform(1, 2, (T, H)) * 2.0 ** np.where(rng.random((T, H)) < 0.8, -1, rng.integers(-spread, 0, (T, H)))
    g = 8.0
    x[:, H - 1] = g  # (in a block of its own: up rows pick the first I)
    xd = torch.from_numpy(x).float().cuda().bfloat16()
    w_up, s = one_hot(wq, I, H)
    w_gate = np.zeros_like(w_up)
    w_gate[..., -1] = 0x38 if wq == "fp8_b128" else (2 if wq == "mxfp4" else 1) << 4
    w_down, s_down = one_hot(wq, H, I)
    dev = lambda a: torch.from_numpy(a.view(np.int16) if a.dtype == np.uint16 else a).cuda()
    d = {k: dev(v) for k, v in dict(w_gate=w_gate, w_up=w_up, w_down=w_down, s_gate=s, s_up=s, s_down=s_down).items()}
    d = {k: v.expand(E, *v.shape[1:]).contiguous() for k, v in d.items()}
    cfg = gb.make_config(T, H, I, E, 1, act="bf16", w=wq)
    assert gb.ffn_kernel(cfg) == ("tc_fp8" if T == 448 else "fm")
    ws, out = workspace(cfg), torch.empty((T, H), dtype=torch.bfloat16, device="cuda")
    gb.moe_forward(cfg, xd, torch.zeros((E, H), dtype=torch.bfloat16, device="cuda"), None, None, wbundle(d), None, out, ws)
    torch.cuda.synchronize()
    assert gb.moe_device_status(ws) == gb.OK
    got, xs = act_np(out), act_np(xd)[:, :I]
    h = g / (1 + np.exp(-g)) * xs
    top = np.abs(h).reshape(T, I // 128, 128).max(-1).repeat(128, axis=1)
    low = 0.0 if spread == 9 else 2.0 ** (-17 if T == 448 else -22)
    worst = np.max(np.abs(got[:, :I] - h) / (2.0**-8 * np.abs(h) + 2 * low * top))
    assert worst <= 1.0, worst
    assert np.all(got[:, I:] == 0)


@pytest.mark.parametrize("wq", CODED)
@pytest.mark.parametrize("e", [13, 24, 30])
@pytest.mark.parametrize("T", [8, 24, 60])
def test_values_beside_an_outlier_keep_their_precision(T, e, wq):
    """One channel in 128 of x is 2^e times the others, one of h (4-bit formats)
    about as much, and every weight is 0 there, so that the output is made of the
    others alone: 16-, 32- and 80-row tiles, with the first pair of codes (2^13) and
    with the second. 1e-2: bf16 rounding of h and y (5e-3 at most over rows of this
    length), and as much again for the codes."""
    wl = BASE.replace(T=T, E=4, top_k=2, H=1024, I=768, wq=wq, seed=T)
    inp = synth.make_inputs(wl)
    inp["x"].reshape(-1, 128)[:, 5] = (127 + e) << 7  # bf16 2^e
    inp["w_router"].reshape(-1, 128)[:, 5] = 0
    ex = inp["experts"]
    for k in ("w_gate", "w_up"):
        if wq == "fp8_b128":
            ex[k][..., 5::128] = 0
        else:
            ex[k][..., 2::64] &= 0x0F  # (the high nibble of byte 2 is channel 5)
    if wq != "fp8_b128":
        for k in ("s_gate", "s_up"):  # rows 9, 137, .. times 2^(e / 2): h there about 2^e times the rest
            ex[k][:, 9::128] += e // 2 + 1 if wq == "mxfp4" else (e // 2 + 1) << 7
        ex["w_down"][..., 4::64] &= 0x0F
    assert_close(act_np(forward(wl, to_device(wl, inp))), oracle.forward(wl, inp)["out"], 1e-2)


@pytest.mark.parametrize("wq", CODED)
@pytest.mark.parametrize("T", [8, 24, 60])
def test_second_codes_of_a_row_leave_the_others_alone(T, wq):
    """Rows that need their second pair of codes make the GEMMs walk k twice; every
    other token's output stays bit for bit as it was."""
    wl = BASE.replace(T=T, E=4, top_k=2, H=1024, I=768, wq=wq, seed=T)
    dev = to_device(wl, synth.make_inputs(wl))
    dev["logit_bias"] = torch.arange(wl.E, device="cuda", dtype=torch.float32) * 1e9  # the routing stays
    a = forward(wl, dev)
    dev["x"][2, 5] = 2.0**30
    dev["x"][5, 700] = -(2.0**24)
    b = forward(wl, dev)
    same = [t for t in range(T) if t not in (2, 5)]
    assert torch.equal(a[same].view(torch.int16), b[same].view(torch.int16))
    assert not torch.equal(a[2].view(torch.int16), b[2].view(torch.int16)) and torch.isfinite(b.float()).all()


def test_mxfp4_scales_at_two_byte_alignment():
    """E8M0 scale tensors need only 2-byte alignment."""
    wl = BASE.replace(T=20, E=8, top_k=2, H=512, I=256, wq="mxfp4", seed=9)
    inp = synth.make_inputs(wl)
    dev = to_device(wl, inp)
    for k in ("s_gate", "s_up", "s_down"):
        v = dev["experts"][k]
        dev["experts"][k] = torch.cat([v.new_zeros(2), v.flatten()])[2:].view(v.shape)
        assert dev["experts"][k].data_ptr() % 4 == 2
    assert_close(act_np(forward(wl, dev)), oracle.forward(wl, inp)["out"], tol(wl))


@pytest.mark.parametrize("T", [8, 40, 120])
def test_mxfp4_weights_at_16_byte_alignment(T):
    """Weights that TMA cannot unpack (it wants 32-byte aligned ones) are decoded
    by the kernel: the same products and scales, so nearly the same output."""
    wl = BASE.replace(T=T, E=4, top_k=2, H=512, I=256, wq="mxfp4", seed=11)
    inp = synth.make_inputs(wl)
    dev = to_device(wl, inp)
    aligned = act_np(forward(wl, dev))
    for k in ("w_gate", "w_up", "w_down"):
        v = dev["experts"][k]
        assert v.data_ptr() % 32 == 0
        dev["experts"][k] = torch.cat([v.flatten()[:16], v.flatten()])[16:].view(v.shape)
        assert dev["experts"][k].data_ptr() % 32 == 16
    got = act_np(forward(wl, dev))
    want = oracle.forward(wl, inp)["out"]
    assert_close(got, want, tol(wl))
    assert_close(aligned, want, tol(wl))


def test_mxfp4_block_scales_far_apart():
    """Scales of one row's four 32-blocks that differ by up to 2^12, and blocks
    2^30 below their neighbours."""
    wl = BASE.replace(T=20, E=4, top_k=2, H=512, I=256, wq="mxfp4", seed=10)
    inp = synth.make_inputs(wl)
    rng = np.random.default_rng(0)
    for k in ("s_gate", "s_up", "s_down"):
        s = inp["experts"][k]
        inp["experts"][k] = (s.astype(np.int32) - rng.integers(0, 13, s.shape)).astype(np.uint8)
        inp["experts"][k][..., ::8, 1] -= 18
    assert_close(act_np(forward(wl, to_device(wl, inp))), oracle.forward(wl, inp)["out"], tol(wl))


@pytest.mark.parametrize("T", [6, 24, 60])
def test_mxfp4_scales_of_each_k_block_are_its_own(T):
    """Scales that step by 2^-3, 2^0 and 2^3 from one 128-wide k block to the
    next, over many k blocks: a block multiplied with the scales of one of the
    blocks whose MMAs are in flight beside it (16-, 32- and 80-row tiles) would
    be off by at least 2^3."""
    wl = BASE.replace(T=T, E=4, top_k=2, H=4096, I=1024, wq="mxfp4", seed=T)
    inp = synth.make_inputs(wl)
    for k in ("s_gate", "s_up", "s_down"):
        s = inp["experts"][k].astype(np.int32)
        step = np.repeat(3 * (np.arange(s.shape[-1] // 4) % 3 - 1), 4)
        inp["experts"][k] = (s + step).astype(np.uint8)
    assert_close(act_np(forward(wl, to_device(wl, inp))), oracle.forward(wl, inp)["out"], tol(wl))


@pytest.mark.parametrize("wq", ["fp8_b128", "int4_g128", "mxfp4"])
@pytest.mark.parametrize("T,I_shared", [(5, 256), (20, 256), (60, 256), (150, 256), (60, 384)])
def test_shared_expert_with_the_routed_ones(T, I_shared, wq):
    """The shared expert runs as one more expert of the same launches when its
    intermediate size is the routed ones', else by itself; 128 routed experts and
    the shared one fill the schedule's warps unevenly."""
    wl = BASE.replace(T=T, E=128, top_k=3, H=512, I=256, wq=wq, seed=T, score="sigmoid", routed_scale=2.5, n_group=4,
                      topk_group=2, has_shared=True, I_shared=I_shared, select_bias_sigma=0.01)
    inp = synth.make_inputs(wl)
    alone = kernel_of(wl) != "fm" or I_shared != wl.I
    assert gb.ffn_kernel(config(wl), shared=True) == (kernel_of(wl.replace(E=1, top_k=1, I=I_shared, has_shared=False)) if alone else "joined")
    assert_close(act_np(forward(wl, to_device(wl, inp), kernel_of(wl))), oracle.forward(wl, inp)["out"], tol(wl, kernel_of(wl)))


def test_shared_expert_after_512_routed_ones():
    wl = BASE.replace(T=40, E=512, top_k=4, H=256, I=128, wq="fp8_b128", seed=3, has_shared=True, I_shared=128)
    inp = synth.make_inputs(wl)
    assert_close(act_np(forward(wl, to_device(wl, inp))), oracle.forward(wl, inp)["out"], tol(wl))


@pytest.mark.parametrize("wq", ["bf16", "fp8_b128", "int4_g128", "mxfp4"])
@pytest.mark.parametrize("T", [24, 120])
def test_bounded_waits_give_up_and_the_next_call_is_clean(T, wq, monkeypatch):
    """With the wait limit lowered to 0 ns every role of the kernel stops, drains
    what it issued and reports; the next call with the normal limit is clean."""
    wl = BASE.replace(T=T, E=8, top_k=2, H=1024, I=512, wq=wq, seed=77)
    inp = synth.make_inputs(wl)
    dev = to_device(wl, inp)
    cfg = config(wl)
    ws = workspace(cfg)
    out = torch.empty((wl.T, wl.H), dtype=torch.bfloat16, device="cuda")
    args = (cfg, dev["x"], dev["w_router"], None, None, wbundle(dev["experts"]), None, out, ws)
    monkeypatch.setenv("GBMOE_TC_WAIT_LIMIT_NS", "0")
    gb.moe_forward(*args)
    assert gb.moe_device_status(ws) == gb.EDEVICE_TIMEOUT
    monkeypatch.delenv("GBMOE_TC_WAIT_LIMIT_NS")
    gb.moe_forward(*args)
    assert gb.moe_device_status(ws) == gb.OK
    assert_close(act_np(out), oracle.forward(wl, inp)["out"], tol(wl))
