"""The work a user of the GTR token mixer has this framework do, as timed cases.

Every case is one call of a public entry point of ``paper_2609_26590_gb300.gla`` on device
tensors: the mixer (``forward`` / ``forward_ws``), the mixer with its output gate
(``forward_gated``), the mixer with its retention gate computed from the rank-16 projection
(``forward_lowrank_gate``) and the Spatial SwiGLU step (``sswiglu_dwconv``).  Sizes are the
repository's own workloads (stride-16 patch grids of 640^2 to 2048^2 images, head widths 32 to
128, batch 1 to 32) and odd ones between them.
"""
import math

import torch

from paper_2609_26590_gb300 import gla

_DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
_ELEM = {"f32": 4, "f16": 2, "bf16": 2}
_RANK = 16  # rank of the retention gate's projection
_EPS = 1e-6


def _mixer(name, op, dtype, B, H, grid_h, grid_w, Dk, Dv, order, tau=16.0, z_mean=0.0, nodecay=0.0,
           final_state=True, prealloc=False):
    c = {"op": op, "dtype": dtype, "B": B, "H": H, "grid_h": grid_h, "grid_w": grid_w, "Dk": Dk, "Dv": Dv,
         "order": order, "tau": tau, "z_mean": z_mean, "nodecay": nodecay, "final_state": final_state,
         "prealloc": prealloc}
    return dict(c, name=name) if name else c


def _swiglu(name, dtype, B, grid_h, grid_w, F, bias=True):
    c = {"op": "sswiglu", "dtype": dtype, "B": B, "grid_h": grid_h, "grid_w": grid_w, "F": F, "bias": bias}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: two heads of a 256^2 image in full precision, as a unit check runs it
        _mixer("mixer_tiny_f32", "mixer", "f32", 1, 2, 16, 16, 64, 64, gla.ROW_FWD),
        # one 640^2 image through a small model's mixer, buffers kept between calls (serving latency)
        _mixer("mixer_b1_640_f16", "mixer", "f16", 1, 6, 40, 40, 64, 64, gla.COL_REV, prealloc=True),
        # 704^2 images: a grid that 64-token chunks do not divide, the narrow-key head shape, no state kept
        _mixer("mixer_704_dk32_bf16", "mixer", "bf16", 8, 12, 44, 44, 32, 64, gla.COL_FWD, final_state=False),
        # a batch of 640^2 images, a tenth of the channels without decay (throughput inference)
        _mixer("mixer_b32_640_bf16", "mixer", "bf16", 32, 12, 40, 40, 64, 64, gla.ROW_FWD, nodecay=0.1),
        # 1280^2 images with strongly decaying gates (6,400 tokens)
        _mixer("mixer_b8_1280_f16", "mixer", "f16", 8, 16, 80, 80, 64, 64, gla.ROW_REV, tau=1.0, z_mean=-1.0),
        # 2048^2 images, 128-wide heads: few, long sequences (16,384 tokens)
        _mixer("mixer_2048_d128_bf16", "mixer", "bf16", 2, 8, 128, 128, 128, 128, gla.COL_FWD),
        # four 640^2 images in full precision (evaluation against a reference)
        _mixer("mixer_b4_640_f32", "mixer", "f32", 4, 6, 40, 40, 64, 64, gla.COL_REV),
        # one 640^2 image, mixer and output gate, buffers kept (a block as it is served)
        _mixer("gated_b1_640_f16", "gated", "f16", 1, 6, 40, 40, 64, 64, gla.ROW_FWD, prealloc=True),
        # the batch with its output gate
        _mixer("gated_b32_640_bf16", "gated", "bf16", 32, 12, 40, 40, 64, 64, gla.ROW_REV, nodecay=0.1),
        # the batch with the retention gate formed from its low-rank projection
        _mixer("lowrank_b32_640_bf16", "lowrank", "bf16", 32, 12, 40, 40, 64, 64, gla.ROW_FWD),
        # one 640^2 image between the projections of a small model's Spatial SwiGLU
        _swiglu("sswiglu_b1_640_f16", "f16", 1, 40, 40, 768),
        # the batch between the projections of the large model's Spatial SwiGLU
        _swiglu("sswiglu_b32_640_bf16", "bf16", 32, 40, 40, 1536),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case of the listed ones' ranges; costs no more than the largest of them."""
    kind = rng.choice(["mixer", "mixer", "mixer", "mixer_f32", "gated", "gated", "lowrank", "lowrank",
                       "sswiglu", "sswiglu"])
    while True:
        if kind == "sswiglu":
            c = _swiglu(None, rng.choice(["f16", "bf16", "f32"]), _log_int(rng, 1, 32), _log_int(rng, 12, 128),
                        _log_int(rng, 12, 128), 8 * _log_int(rng, 8, 288), rng.random() < 0.7)
            if 1e6 <= work(c)["bytes"] <= 4.5e8:
                return c
            continue
        f32 = kind == "mixer_f32"
        B, H = _log_int(rng, 1, 32), _log_int(rng, 2, 16)
        gh, gw = (_log_int(rng, 12, 40), _log_int(rng, 12, 40)) if f32 else (_log_int(rng, 16, 128), _log_int(rng, 16, 128))
        Dk = rng.choice([32, 64, 64, 64] if kind == "lowrank" else [32, 40, 64, 64, 64, 96, 128])
        Dv = rng.choice([64, 64, 64, 128]) if Dk <= 64 else rng.choice([64, 128])
        tau, z_mean = rng.choice([(16.0, 0.0), (16.0, 0.0), (1.0, -1.0)])
        c = _mixer(None, "mixer" if f32 else kind, "f32" if f32 else rng.choice(["f16", "bf16"]), B, H, gh, gw, Dk, Dv,
                   rng.randrange(4), tau, z_mean, 0.0 if kind == "lowrank" else rng.choice([0.0, 0.1]),
                   rng.random() < 0.5, rng.random() < 0.3 and kind != "lowrank")
        # full precision: at most the listed evaluation's sequences; 16 bits: half the batch's bytes
        # (the narrower and wider heads take longer per byte)
        if f32 and B * H > 24:
            continue
        if 4e5 <= work(c)["bytes"] <= 2e8:
            return c


def _gates(shape, tau, z_mean, nodecay, gen):
    z = torch.randn(shape, device="cuda", generator=gen) + z_mean
    g = torch.nn.functional.logsigmoid(z) / tau
    if nodecay > 0.0:  # a share of the (head, key channel) pairs never forgets
        n = shape[2] * shape[3]
        sel = torch.randperm(n, device="cuda", generator=gen)[: int(round(nodecay * n))]
        keep = torch.ones(n, device="cuda")
        keep[sel] = 0.0
        g = g * keep.view(shape[2], shape[3])
    return g


def _inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    dt = _DTYPES[case["dtype"]]

    def randn(*shape):
        return torch.randn(shape, device="cuda", generator=gen)

    if case["op"] == "sswiglu":
        B, T, F = case["B"], case["grid_h"] * case["grid_w"], case["F"]
        return {"h": randn(B, T, 2 * F).to(dt), "weight": randn(F, 3, 3) / 3.0,
                "bias": 0.1 * randn(F) if case["bias"] else None}
    B, H, Dk, Dv = case["B"], case["H"], case["Dk"], case["Dv"]
    T = case["grid_h"] * case["grid_w"]
    x = {"q": randn(B, T, H, Dk).to(dt), "k": (randn(B, T, H, Dk) / math.sqrt(Dk)).to(dt), "v": randn(B, T, H, Dv).to(dt)}
    if case["op"] == "lowrank":
        x["a"] = randn(B, T, _RANK).to(dt)
        x["w2"] = (randn(H, _RANK, Dk) / math.sqrt(_RANK)).to(dt)
        x["gate_bias"] = case["z_mean"] + 0.25 * randn(H, Dk)
    else:
        x["g"] = _gates((B, T, H, Dk), case["tau"], case["z_mean"], case["nodecay"], gen).to(dt)
    if case["op"] == "gated":
        x["r"] = randn(B, T, H, Dv).to(dt)
        x["norm_weight"] = 1.0 + 0.1 * randn(Dv)
    return x


def prepare(case, seed):
    s = dict(case, x=_inputs(case, seed))
    x = s["x"]
    if case["op"] == "sswiglu":
        s["gate"], s["value"] = x["h"][..., : case["F"]], x["h"][..., case["F"]:]
        return s
    s["out"] = s["fs"] = s["ws"] = None
    if case["prealloc"]:  # a serving loop's own buffers
        B, H, Dk, Dv = case["B"], case["H"], case["Dk"], case["Dv"]
        s["out"] = torch.empty_like(x["v"])
        if case["final_state"]:
            s["fs"] = torch.empty((B, H, Dk, Dv), dtype=torch.float32, device="cuda")
        n = gla.workspace_bytes(B, H, case["grid_h"], case["grid_w"], Dk, Dv, x["q"].dtype)
        s["ws"] = torch.empty(max(n, 256), dtype=torch.uint8, device="cuda")
    return s


def run(s):
    x, gh, gw = s["x"], s["grid_h"], s["grid_w"]
    if s["op"] == "sswiglu":
        return gla.sswiglu_dwconv(s["gate"], s["value"], x["weight"], x["bias"], gh, gw)
    fs = s["fs"] if s["prealloc"] else s["final_state"]
    if s["op"] == "mixer":
        if s["prealloc"]:
            gla.forward_ws(x["q"], x["k"], x["v"], x["g"], gh, gw, s["order"], s["out"], fs, s["ws"])
            return s["out"], fs
        return gla.forward(x["q"], x["k"], x["v"], x["g"], gh, gw, s["order"], final_state=fs)
    if s["op"] == "gated":
        return gla.forward_gated(x["q"], x["k"], x["v"], x["g"], x["r"], x["norm_weight"], _EPS, gh, gw, s["order"],
                                 out=s["out"], final_state=fs, workspace=s["ws"])
    return gla.forward_lowrank_gate(x["q"], x["k"], x["v"], x["a"], x["w2"], x["gate_bias"], s["tau"], gh, gw,
                                    s["order"], final_state=fs)


def work(case):
    es = _ELEM[case["dtype"]]
    if case["op"] == "sswiglu":
        n, F = case["B"] * case["grid_h"] * case["grid_w"], case["F"]
        return {"bytes": 3.0 * n * F * es + (10 if case["bias"] else 9) * F * 4, "flops": 24.0 * n * F}
    B, H, Dk, Dv = case["B"], case["H"], case["Dk"], case["Dv"]
    n = B * case["grid_h"] * case["grid_w"] * H
    if case["op"] == "lowrank":
        nbytes = n * es * (2 * Dk + 2 * Dv) + n // H * _RANK * es + H * Dk * (_RANK * es + 4)
    else:
        nbytes = n * es * (3 * Dk + 2 * Dv)
    if case["op"] == "gated":
        nbytes += n * es * Dv + 4 * Dv
    if case["final_state"]:
        nbytes += 4 * B * H * Dk * Dv
    # summaries and readout, the causal triangle of 64-token chunks, the state's decay
    flops = n * (4.0 * Dk * Dv + 65.0 * (Dk + Dv) + Dk * Dv / 32.0)
    if case["op"] == "lowrank":
        flops += 2.0 * n * _RANK * Dk
    return {"bytes": float(nbytes), "flops": flops}


def exact(case, seed):
    x = {n: t.double() if t is not None else None for n, t in _inputs(case, seed).items()}
    gh, gw, B = case["grid_h"], case["grid_w"], case["B"]
    T = gh * gw
    if case["op"] == "sswiglu":
        F = case["F"]
        gate, value = x["h"][..., :F], x["h"][..., F:].reshape(B, gh, gw, F)
        pad = torch.nn.functional.pad(value, (0, 0, 1, 1, 1, 1))
        acc = torch.zeros_like(value) if x["bias"] is None else x["bias"].expand(B, gh, gw, F).clone()
        for i in range(3):
            for j in range(3):
                acc += x["weight"][:, i, j] * pad[:, i:i + gh, j:j + gw]
        return gate * torch.sigmoid(gate) * acc.view(B, T, F)
    H, Dk, Dv = case["H"], case["Dk"], case["Dv"]
    q, k, v = x["q"], x["k"], x["v"]
    if case["op"] == "lowrank":
        z = torch.einsum("btr,hrd->bthd", x["a"], x["w2"]) + x["gate_bias"]
        g = torch.nn.functional.logsigmoid(z) / case["tau"]
    else:
        g = x["g"]
    s = torch.arange(T, device="cuda")
    u = T - 1 - s if case["order"] in (gla.ROW_REV, gla.COL_REV) else s
    tok = u if case["order"] in (gla.ROW_FWD, gla.ROW_REV) else (u % gh) * gw + u // gh
    # S_t = Diag(e^{g_t}) S_{t-1} + k_t^T v_t, o_t = q_t S_t, in blocks of C tokens
    C, N = 16, B * H
    S = torch.zeros((N, Dk, Dv), dtype=torch.float64, device="cuda")
    o = torch.empty((B, T, H, Dv), dtype=torch.float64, device="cuda")
    for s0 in range(0, T, C):
        t = tok[s0:s0 + C]
        n = t.numel()
        qc, kc, vc, gc = (y[:, t].transpose(1, 2).reshape(N, n, -1) for y in (q, k, v, g))
        A = gc.cumsum(1)
        later = torch.ones(n, n, dtype=torch.bool, device="cuda").triu(1)
        P = torch.empty((N, n, n), dtype=torch.float64, device="cuda")
        for j in range(n):  # scores of key j for every query at or after it
            P[:, :, j] = (qc * kc[:, j:j + 1] * torch.exp((A - A[:, j:j + 1]).clamp(max=0.0))).sum(-1)
        P.masked_fill_(later, 0.0)
        oc = torch.bmm(qc * torch.exp(A), S) + torch.bmm(P, vc)
        o[:, t] = oc.view(B, H, n, Dv).transpose(1, 2)
        last = A[:, -1:]
        S = torch.exp(last).transpose(1, 2) * S + torch.bmm((kc * torch.exp(last - A)).transpose(1, 2), vc)
    if case["op"] == "gated":
        r = x["r"]
        o = r * torch.sigmoid(r) * o * torch.rsqrt(o.square().mean(-1, keepdim=True) + _EPS) * x["norm_weight"]
    return o, S.view(B, H, Dk, Dv) if case["final_state"] else None
