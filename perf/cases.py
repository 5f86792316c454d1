"""What the speed of this framework is measured on: whole MoE layer forwards
(moe_forward) as a serving program makes them, from one token to a large
prefill batch, over every expert-weight format and both activation types.

The shapes are those of the repository's own benchmark workloads (tiny fp32,
bf16 with 128 experts, DeepSeek-style fp8 and MXFP4 with 256 experts and a
shared one, skewed int4), each at a decode-sized and a prefill-sized batch;
draw() spreads sizes, types and batches over the ranges between them. Weights
are N(0, 0.02) in their storage format, activations N(0, 1), as in the
benchmark. Every case leaves all routes to AUTO, as a user does.
"""
import math

import torch

import paper_2607_12875_gb300 as gb

DEV = "cuda"
SIGMA_W = 0.02
SIGMA_BIAS = 0.01     # DeepSeek-style selection bias
CHUNK = 1 << 26       # weight elements generated at a time


def _case(name, T, H, I, E, top_k, act="bf16", w="bf16", deepseek=False, skew=0.0, routing=False):
    """deepseek: sigmoid scores, 8 expert groups of which 4 are kept, weights
    times 2.5, selection bias and one shared expert of the same size.
    skew: logit offsets -skew * ln(e + 1), a hot-to-cold order of the experts.
    routing: the caller also asks for the chosen experts, their weights and the
    rows per expert (for load statistics)."""
    c = dict(T=T, H=H, I=I, E=E, top_k=top_k, act=act, w=w, deepseek=deepseek, skew=skew, routing=routing)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest layer a test or a toy model runs: launches and latency only
        _case("tiny_f32_T64", 64, 256, 512, 8, 2, act="f32", w="f32", routing=True),
        # a full-precision run of a small model's batch (odd token count): fp32 on CUDA cores
        _case("batch_f32_T1001", 1001, 1024, 768, 16, 4, act="f32", w="f32"),
        # one sequence being decoded: eight experts' weights, every launch's latency shows
        _case("decode_bf16_T1", 1, 4096, 1536, 128, 8),
        # the headline: a decode batch of 32 sequences
        _case("decode_bf16_T32", 32, 4096, 1536, 128, 8),
        # a larger decode batch or a prompt chunk, odd size: about 20 rows per expert
        _case("chunk_bf16_T333", 333, 4096, 1536, 128, 8),
        # prefill of long prompts: about 512 rows per expert
        _case("prefill_bf16_T8192", 8192, 4096, 1536, 128, 8),
        # DeepSeek-style block-fp8 layer, decode batch and prefill chunk
        _case("decode_fp8_T48", 48, 7168, 2048, 256, 8, w="fp8_b128", deepseek=True),
        _case("prefill_fp8_T2048", 2048, 7168, 2048, 256, 8, w="fp8_b128", deepseek=True, routing=True),
        # int4 experts with skewed routing, decode batch and the largest prefill
        _case("decode_int4_T17", 17, 4096, 2816, 64, 6, w="int4_g128", skew=0.6222),
        _case("prefill_int4_T16384", 16384, 4096, 2816, 64, 6, w="int4_g128", skew=0.6222),
        # the DeepSeek-style layer with MXFP4 experts, small decode batch and prefill chunk
        _case("decode_mxfp4_T16", 16, 7168, 2048, 256, 8, w="mxfp4", deepseek=True),
        _case("prefill_mxfp4_T2048", 2048, 7168, 2048, 256, 8, w="mxfp4", deepseek=True),
    ]


def draw(rng):
    """A layer of one of the families above with other sizes: tokens spread over
    their logarithm, hidden and intermediate sizes over the multiples of 256 and
    128 that the layer takes."""
    def tokens(most):
        return max(1, min(most, round(math.exp(rng.uniform(0.0, math.log(most + 0.5))))))

    def mult(lo, hi, step):
        return step * rng.randint(lo // step, hi // step)

    w = rng.choice(["f32", "bf16", "bf16", "fp8_b128", "int4_g128", "mxfp4"])
    routing = rng.random() < 0.25
    if w == "f32":
        return _case(None, tokens(1500), mult(256, 1024, 256), mult(128, 768, 128), rng.randint(2, 24), 2, act="f32",
                     w="f32", routing=routing)
    if w == "bf16":
        return _case(None, tokens(8192), mult(1024, 4096, 256), mult(512, 1536, 128), rng.randint(16, 128),
                     rng.randint(2, 8), routing=routing)
    if w == "int4_g128":
        return _case(None, tokens(16384), mult(1024, 4096, 256), mult(512, 2816, 128), rng.randint(12, 64),
                     rng.randint(2, 6), w=w, skew=rng.choice([0.0, 0.3, 0.6]), routing=routing)
    return _case(None, tokens(2048), mult(2048, 7168, 256), mult(512, 2048, 128), 8 * rng.randint(8, 32), 8, w=w,
                 deepseek=True, routing=routing)


# ---------------------------------------------------------------- inputs


def _stored(g, w, E, N, K):
    """[E, N, K] weights ~ N(0, SIGMA_W) in the storage format w: (codes, scales or None)."""
    if w in ("f32", "bf16"):
        out = torch.empty((E, N, K), dtype=torch.float32 if w == "f32" else torch.bfloat16, device=DEV)
        return out.normal_(0.0, SIGMA_W, generator=g), None
    packed = w in ("int4_g128", "mxfp4")
    q = torch.empty((E, N, K // 2 if packed else K), dtype=torch.uint8, device=DEV)
    if w == "fp8_b128":
        s = torch.empty((E, N // 128, K // 128), dtype=torch.float32, device=DEV)
    elif w == "int4_g128":
        s = torch.empty((E, N, K // 128), dtype=torch.bfloat16, device=DEV)
    else:
        s = torch.empty((E, N, K // 32), dtype=torch.uint8, device=DEV)
    step = max(1, CHUNK // (N * K))
    for e in range(0, E, step):
        n = min(step, E - e)
        v = torch.empty((n, N, K), device=DEV).normal_(0.0, SIGMA_W, generator=g)
        if w == "fp8_b128":  # one scale per 128 x 128 block
            b = v.view(n, N // 128, 128, K // 128, 128)
            sc = b.abs().amax(dim=(2, 4)) / 448.0
            s[e:e + n] = sc
            q[e:e + n] = (b / sc[:, :, None, :, None]).view(n, N, K).to(torch.float8_e4m3fn).view(torch.uint8)
            continue
        if w == "int4_g128":  # one scale per 128 of a row
            b = v.view(n, N, K // 128, 128)
            sc = (b.abs().amax(-1) / 7.0).to(torch.bfloat16)
            s[e:e + n] = sc
            c = (b / sc.float()[..., None]).round_().clamp_(-8, 7).to(torch.int8).view(torch.uint8) & 15
        else:  # MXFP4: a power-of-two scale per 32 of a row, E2M1 codes (round to even)
            b = v.view(n, N, K // 32, 32)
            ex = torch.floor(torch.log2(b.abs().amax(-1))) - 2.0
            s[e:e + n] = (ex + 127.0).to(torch.uint8)
            a = b.abs() * torch.exp2(-ex)[..., None]
            m = torch.where(a < 2, (2 * a).round(), torch.where(a < 4, a.round() + 2, (a / 2).round() + 4)).clamp_(max=7)
            c = m.to(torch.uint8) | ((b < 0).to(torch.uint8) << 3)
        c = c.view(n, N, K // 2, 2)
        q[e:e + n] = c[..., 0] | (c[..., 1] << 4)
    return q, s


def _experts(g, case, E):
    H, I = case["H"], case["I"]
    d = {}
    for name, N, K in (("gate", I, H), ("up", I, H), ("down", H, I)):
        d["w_" + name], d["s_" + name] = _stored(g, case["w"], E, N, K)
    return d


def _inputs(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    act = torch.float32 if case["act"] == "f32" else torch.bfloat16
    T, H, E = case["T"], case["H"], case["E"]
    d = {"x": torch.empty((T, H), device=DEV).normal_(0.0, 1.0, generator=g).to(act),
         "w_router": torch.empty((E, H), device=DEV).normal_(0.0, SIGMA_W, generator=g).to(act),
         "logit_bias": None, "select_bias": None, "shared": None}
    if case["skew"]:
        d["logit_bias"] = -case["skew"] * torch.log(torch.arange(1, E + 1, device=DEV, dtype=torch.float32))
    if case["deepseek"]:
        d["select_bias"] = torch.empty(E, device=DEV).normal_(0.0, SIGMA_BIAS, generator=g)
        d["shared"] = _experts(g, case, 1)
    d["experts"] = _experts(g, case, E)
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    ds = case["deepseek"]
    cfg = gb.make_config(case["T"], case["H"], case["I"], case["E"], case["top_k"],
                         score="sigmoid" if ds else "softmax", n_group=8 if ds else 1, topk_group=4 if ds else 1,
                         routed_scale=2.5 if ds else 1.0, act=case["act"], w=case["w"], has_shared=ds,
                         I_shared=case["I"] if ds else 0)

    def bundle(w):
        return w and gb.weights(w["w_gate"], w["w_up"], w["w_down"], w["s_gate"], w["s_up"], w["s_down"])

    d["cfg"], d["w_experts"], d["w_shared"] = cfg, bundle(d["experts"]), bundle(d["shared"])
    d["ws"] = torch.empty(gb.workspace_size(cfg), dtype=torch.uint8, device=DEV)
    d["out"] = torch.empty_like(d["x"])
    pairs = (case["T"], case["top_k"])
    d["topk_ids"] = torch.empty(pairs, dtype=torch.int32, device=DEV) if case["routing"] else None
    d["topk_w"] = torch.empty(pairs, dtype=torch.float32, device=DEV) if case["routing"] else None
    d["counts"] = torch.empty(case["E"], dtype=torch.int32, device=DEV) if case["routing"] else None
    return d


def run(s):
    gb.moe_forward(s["cfg"], s["x"], s["w_router"], s["logit_bias"], s["select_bias"], s["w_experts"], s["w_shared"],
                   s["out"], s["ws"], topk_ids=s["topk_ids"], topk_w=s["topk_w"], counts=s["counts"])
    return {k: s[k] for k in ("out", "topk_ids", "topk_w", "counts") if s[k] is not None}


# ------------------------------------------------- work, tolerance, 64 bits


def _expert_bytes(case):
    n = 3 * case["H"] * case["I"]
    return {"f32": 4 * n, "bf16": 2 * n, "fp8_b128": n + 4 * n // 16384, "int4_g128": n // 2 + 2 * n // 128,
            "mxfp4": n // 2 + n // 32}[case["w"]]


def work(case):
    """Every expert that receives rows read once (their expected number under
    even routing), activations in and out once; two operations per product."""
    T, H, I, E, k = case["T"], case["H"], case["I"], case["E"], case["top_k"]
    a = 4 if case["act"] == "f32" else 2
    active = E * (1.0 - (1.0 - k / E) ** T)
    shared = 1 if case["deepseek"] else 0
    return {"bytes": (active + shared) * _expert_bytes(case) + a * H * (2 * T + E),
            "flops": 2.0 * T * H * E + 6.0 * T * (k + shared) * H * I}


def tolerance(case):
    """About four times what a forward differs from the 64-bit one: fp32 sums,
    or bf16 intermediates and results (2e-3 to 4e-3)."""
    return {"rel": 1e-5} if case["act"] == "f32" else {"rel": 1.2e-2}


_E2M1 = (0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 6.0, -0.0, -0.5, -1.0, -1.5, -2.0, -3.0, -4.0, -6.0)


def _wide(w, q, s, e):
    """Expert e's matrix in 64 bits."""
    if s is None:
        return q[e].double()
    if w == "fp8_b128":
        sc = s[e].double().repeat_interleave(128, 0).repeat_interleave(128, 1)
        return q[e].view(torch.float8_e4m3fn).float().double() * sc
    c = torch.stack((q[e] & 15, q[e] >> 4), -1).view(q.shape[1], -1).long()
    if w == "int4_g128":
        return (c - 16 * (c >= 8)).double() * s[e].double().repeat_interleave(128, 1)
    table = torch.tensor(_E2M1, dtype=torch.float64, device=DEV)
    return table[c] * torch.exp2(s[e].double() - 127.0).repeat_interleave(32, 1)


def _ffn(case, d, e, x):
    def mat(n):
        return _wide(case["w"], d["w_" + n], d["s_" + n], e)
    return (torch.nn.functional.silu(x @ mat("gate").T) * (x @ mat("up").T)) @ mat("down").T


def exact(case, seed):
    d = _inputs(case, seed)
    T, E, k = case["T"], case["E"], case["top_k"]
    x = d["x"].double()
    logits = x @ d["w_router"].double().T
    if d["logit_bias"] is not None:
        logits = logits + d["logit_bias"].double()
    if case["deepseek"]:
        score = torch.sigmoid(logits)
        key = score + d["select_bias"].double()
        grp = key.view(T, 8, E // 8).topk(2, dim=-1).values.sum(-1)
        keep = torch.zeros_like(grp, dtype=torch.bool).scatter_(1, grp.topk(4, dim=-1).indices, True)
        key = key.masked_fill(~keep.repeat_interleave(E // 8, 1), -math.inf)
        ids = key.topk(k, dim=-1).indices
        wt = score.gather(1, ids)
        wt = 2.5 * wt / wt.sum(-1, keepdim=True)
    else:
        top = logits.topk(k, dim=-1)
        ids, wt = top.indices, torch.softmax(top.values, -1)
    out = torch.zeros_like(x)
    for e in range(E):
        t, j = torch.nonzero(ids == e, as_tuple=True)
        if t.numel():
            out.index_add_(0, t, wt[t, j][:, None] * _ffn(case, d["experts"], e, x[t]))
    if d["shared"] is not None:
        out += _ffn(case, d["shared"], 0, x)
    full = {"out": out, "topk_ids": None, "topk_w": wt, "counts": None}
    return full if case["routing"] else {"out": out}
