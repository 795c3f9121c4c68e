"""Performance cases: the calls that users of the library make, over the sizes it is used at.

``listed()`` are the named cases, ``draw(rng)`` gives further ones of the same
ranges. ``prepare`` makes what a program has in hand before the call (inputs,
Lambda or the layer's weights, output buffers, the workspace), ``run`` makes
the call or calls of one pass through the public entry points and returns
their outputs, ``work`` counts the bytes and operations a pass cannot do
without, ``exact`` evaluates the same outputs in float64 with plain torch.

Kinds of cases:
  scan   blr_scan_fwd (+ blr_scan_bwd when "train"), in its plain, gated and
         varlen forms; x, h, dh: (B, L, D), gate logits (B, L, 2D)
  step   blr_step: one recurrent-inference step of B states
  steps  blr_steps: K steps of B states, every state returned
  layer  one forward and backward of the gated recurrent layer
"""
import math

import torch

import paper_2406_12580_gb300 as blr
from paper_2406_12580_gb300.layer import GatedRecurrentLayer

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}
CODES = {"f32": blr.BLR_F32, "bf16": blr.BLR_BF16}
MAX_BYTES = 3.8e9  # what the largest listed case moves


def _scan(io, B, L, D, mode="plain", train=True, state=False, lo=0.9, hi=0.999, c=1.0, pad=0.0,
          gate_std=1.0):
    """state: the program passes h0 and dh_last and takes dh0; pad: share of leading zero rows."""
    return dict(kind="scan", io=io, B=B, L=L, D=D, mode=mode, train=train, state=state, lo=lo,
                hi=hi, c=c, pad=pad, gate_std=gate_std)


def listed():
    return [
        # scoring a handful of users with histories of the short datasets' maximum length
        dict(name="infer_4x50x64_f32", **_scan("f32", 4, 50, 64, train=False)),
        # a training step's scan at the maximum length of ML-1M, float32
        dict(name="train_256x200x64_f32", **_scan("f32", 256, 200, 64)),
        # the paper's training batch in bfloat16, left-padded, as the layer calls it (merge fused)
        dict(name="gated_2048x50x64_bf16",
             **_scan("bf16", 2048, 50, 64, mode="gated", pad=0.2, gate_std=0.5)),
        # the same kind of batch with the rows' own lengths instead of padding
        dict(name="varlen_1000x200x64_bf16", **_scan("bf16", 1000, 200, 64, mode="varlen")),
        # long user histories (XLong), many rows, float32
        dict(name="train_64x2048x256_f32", **_scan("f32", 64, 2048, 256, lo=0.99, hi=0.9999)),
        # few users with medium histories, odd sizes, resumed from a state
        dict(name="train_12x1031x200_bf16", **_scan("bf16", 12, 1031, 200, state=True)),
        # few long sequences in float32
        dict(name="train_8x8192x512_f32", **_scan("f32", 8, 8192, 512, lo=0.99, hi=0.9999)),
        # few very long sequences in bfloat16: the scan by itself, and with the layer's merge
        dict(name="train_8x32768x512_bf16", **_scan("bf16", 8, 32768, 512, lo=0.99, hi=0.9999)),
        dict(name="gated_8x32768x512_bf16",
             **_scan("bf16", 8, 32768, 512, mode="gated", lo=0.99, hi=0.9999)),
        # serving: one new behavior of every active user, and eight at once
        dict(name="step_65536x64_f32", kind="step", io="f32", B=65536, D=64, c=1.0),
        dict(name="steps_65536x8x64_bf16", kind="steps", io="bf16", B=65536, K=8, D=64, c=1.0),
        # a whole gated recurrent layer, forward and backward, float32
        dict(name="layer_256x200x64_f32", kind="layer", B=256, L=200, d_model=64, expand=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["scan"] * 7 + ["step", "steps", "layer"])
    io = rng.choice(["f32", "bf16"])
    if kind == "layer":
        return dict(kind="layer", B=_log_int(rng, 4, 512), L=_log_int(rng, 20, 200),
                    d_model=8 * rng.randint(2, 16), expand=rng.choice([1, 2]))
    if kind in ("step", "steps"):
        D = 8 * _log_int(rng, 2, 32)
        B = _log_int(rng, 16, 65536 * 64 // D)
        c = rng.choice([1.0, 1.0, 8.0])
        if kind == "step":
            return dict(kind="step", io=io, B=B, D=D, c=c)
        return dict(kind="steps", io=io, B=B, K=rng.randint(2, 12), D=D, c=c)
    mode = rng.choice(["plain", "plain", "gated", "gated", "varlen"])
    train = rng.random() < 0.75
    while True:
        L = _log_int(rng, 20, 32768)
        B = _log_int(rng, 1, 2048)
        D = 8 * _log_int(rng, 1, 64)
        c = _scan(io, B, L, D, mode=mode, train=train, state=rng.random() < 0.4,
                  lo=rng.choice([0.9, 0.99]), hi=rng.choice([0.999, 0.9999]),
                  c=rng.choice([1.0, 1.0, 1.0, 8.0]))
        if B * L * D >= 4096 and work(c)["bytes"] <= MAX_BYTES / 2:
            return c


# ------------------------------------------------------------------ inputs


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _normal(g, shape, dtype, std=1.0):
    return (torch.randn(shape, generator=g, device="cuda", dtype=torch.float32) * std).to(dtype)


def _lambda(g, D, lo, hi):
    """exp(-softplus(Lambda)) uniform in [lo, hi]."""
    u = torch.rand(D, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo
    return torch.log((1.0 - u) / u).float()


def _scan_inputs(case, seed):
    g = _generator(seed)
    B, L, D, T = case["B"], case["L"], case["D"], DTYPES[case["io"]]
    s = {"lam": _lambda(g, D, case["lo"], case["hi"])}
    s["x"] = _normal(g, (B, L, D), T)
    s["gl"] = _normal(g, (B, L, 2 * D), T, case["gate_std"])
    s["z"] = _normal(g, (B, L, D), T) if case["mode"] == "gated" else None
    s["dh"] = _normal(g, (B, L, D), T) if case["train"] else None
    s["h0"] = _normal(g, (B, D), torch.float32) if case["state"] else None
    s["dh_last"] = _normal(g, (B, D), torch.float32) if case["state"] and case["train"] else None
    s["lengths"] = None
    if case["mode"] == "varlen":
        s["lengths"] = torch.randint(1, L + 1, (B,), generator=g, device="cuda", dtype=torch.int32)
    p = int(case["pad"] * L)
    if p > 0:
        s["x"][:, :p] = 0
        s["gl"][:, :p] = 0
    return s


def _step_inputs(case, seed):
    g = _generator(seed)
    B, D, T = case["B"], case["D"], DTYPES[case["io"]]
    S = torch.float32 if case["kind"] == "step" else T
    K = () if case["kind"] == "step" else (case["K"],)
    return {"lam": _lambda(g, D, 0.99, 0.9999), "h": _normal(g, (B, D), S),
            "x": _normal(g, (B, *K, D), T), "gl": _normal(g, (B, *K, 2 * D), T)}


LAYER_PARAMS = ("in_proj.weight", "in_proj.bias", "conv.weight", "conv.bias", "gate_proj.weight",
                "gate_proj.bias", "lam", "out_proj.weight", "out_proj.bias")


def _layer_inputs(case, seed):
    g = _generator(seed)
    d, ed, W = case["d_model"], case["expand"] * case["d_model"], 4

    def uniform(shape, fan):
        return (torch.rand(shape, generator=g, device="cuda") * 2 - 1) / math.sqrt(fan)

    p = {"in_proj.weight": uniform((2 * ed, d), d), "in_proj.bias": uniform((2 * ed,), d),
         "conv.weight": uniform((ed, 1, W), W), "conv.bias": uniform((ed,), W),
         "gate_proj.weight": uniform((2 * ed, ed), ed), "gate_proj.bias": uniform((2 * ed,), ed),
         "lam": _lambda(g, ed, 0.9, 0.999),
         "out_proj.weight": uniform((d, ed), ed), "out_proj.bias": uniform((d,), ed)}
    h = _normal(g, (case["B"], case["L"], d), torch.float32)
    dy = _normal(g, (case["B"], case["L"], d), torch.float32)
    return p, h, dy


def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "layer":
        p, h, dy = _layer_inputs(case, seed)
        layer = GatedRecurrentLayer(case["d_model"], case["expand"], 4, device="cuda")
        with torch.no_grad():
            for name, q in layer.named_parameters():
                q.copy_(p[name])
        params = dict(layer.named_parameters())
        s.update(layer=layer, params=[params[n] for n in LAYER_PARAMS], h=h.requires_grad_(), dy=dy)
        return s
    if case["kind"] in ("step", "steps"):
        s.update(_step_inputs(case, seed))
        s["h_out"] = torch.empty_like(s["h"])
        s["h_seq"] = torch.empty_like(s["x"]) if case["kind"] == "steps" else None
        return s
    s.update(_scan_inputs(case, seed))
    B, L, D = case["B"], case["L"], case["D"]
    s["desc"] = blr.Desc(B, L, D, CODES[case["io"]], case["c"])
    # rows before a sequence's start are not written: they stay zero
    new = torch.zeros_like if case["mode"] == "varlen" else torch.empty_like
    s["y"] = new(s["x"])
    s["h_last"] = torch.empty(B, D, dtype=torch.float32, device="cuda")
    s["ws"] = torch.empty(blr.blr_workspace_bytes(s["desc"]), dtype=torch.uint8, device="cuda")
    if case["train"]:
        s["dx"], s["dgl"] = new(s["x"]), new(s["gl"])
        s["dz"] = new(s["z"]) if s["z"] is not None else None
        s["dlam"] = torch.empty_like(s["lam"])
        s["dh0"] = torch.empty_like(s["h_last"]) if case["state"] else None
    return s


# --------------------------------------------------------------------- run


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "layer":
        y = s["layer"](s["h"])
        return (y, *torch.autograd.grad(y, [s["h"], *s["params"]], s["dy"]))
    if kind == "step":
        blr.blr_step(case["B"], case["D"], CODES[case["io"]], case["c"], s["h"], s["x"], s["gl"],
                     s["lam"], s["h_out"])
        return {"h": s["h_out"]}
    if kind == "steps":
        code = CODES[case["io"]]
        blr.blr_steps(case["B"], case["K"], case["D"], code, code, case["c"], s["h"], s["x"],
                      s["gl"], s["lam"], s["h_out"], s["h_seq"])
        return {"h": s["h_out"], "h_seq": s["h_seq"]}
    mode, desc, out = case["mode"], s["desc"], {"y": s["y"], "h_last": s["h_last"]}
    if mode == "plain":
        blr.blr_scan_fwd(desc, s["x"], s["gl"], s["lam"], s["h0"], s["y"], s["h_last"], s["ws"])
    elif mode == "gated":
        blr.blr_scan_fwd_gated(desc, s["x"], s["gl"], s["lam"], s["h0"], s["z"], s["y"],
                               s["h_last"], s["ws"])
    else:
        blr.blr_scan_fwd_varlen(desc, s["lengths"], s["x"], s["gl"], s["lam"], s["h0"], s["y"],
                                s["h_last"], s["ws"])
    if not case["train"]:
        return out
    grads = {k: s[k] for k in ("dx", "dgl", "dz", "dlam", "dh0") if s[k] is not None}
    if mode == "plain":
        blr.blr_scan_bwd(desc, s["dh"], s["dh_last"], s["x"], s["gl"], s["lam"], s["h0"], s["dx"],
                         s["dgl"], s["dlam"], s["dh0"], s["ws"])
    elif mode == "gated":
        blr.blr_scan_bwd_gated(desc, s["dh"], s["dh_last"], s["x"], s["gl"], s["lam"], s["h0"],
                               s["z"], s["dx"], s["dgl"], s["dz"], s["dlam"], s["dh0"], s["ws"])
    else:
        blr.blr_scan_bwd_varlen(desc, s["lengths"], s["dh"], s["dh_last"], s["x"], s["gl"],
                                s["lam"], s["h0"], s["dx"], s["dgl"], s["dlam"], s["dh0"],
                                s["ws"])
    return {**out, **grads}


# -------------------------------------------------------------------- work


def work(case):
    """Bytes: every input read once, every output written once. Operations: the
    arithmetic of the definitions (a sigmoid, exponential or square root as one)."""
    kind = case["kind"]
    if kind == "layer":
        d, ed, T = case["d_model"], case["expand"] * case["d_model"], case["B"] * case["L"]
        weights = 2 * ed * d + 2 * ed * ed + ed * d + 4 * ed + 7 * ed + d
        gemm = 2 * T * (2 * ed * d + 2 * ed * ed + ed * d)
        return {"bytes": 4.0 * (4 * T * d + 2 * weights), "flops": 3.0 * gemm + 80.0 * T * ed}
    es = 4 if case["io"] == "f32" else 2
    if kind == "step":
        n = case["B"] * case["D"]
        return {"bytes": n * (8.0 + 3 * es) + 4.0 * case["D"], "flops": 12.0 * n}
    if kind == "steps":
        n = case["B"] * case["D"]
        return {"bytes": float(es) * n * (2 + 4 * case["K"]) + 4.0 * case["D"],
                "flops": 12.0 * n * case["K"]}
    n, bd = case["B"] * case["L"] * case["D"], case["B"] * case["D"]
    if case["mode"] == "varlen":  # lengths are uniform in [1, L]
        n *= (case["L"] + 1) / (2 * case["L"])
    gated, state = case["mode"] == "gated", case["state"]
    b = es * n * (5 if gated else 4) + 4.0 * bd * (1 + state) + 4.0 * case["D"]
    f = n * (16 if gated else 12)
    if case["train"]:
        b += es * n * (9 if gated else 7) + 4.0 * bd * 3 * state + 8.0 * case["D"]
        f += n * (40 if gated else 30)
    return {"bytes": float(b), "flops": float(f)}


# ------------------------------------------------------------------- exact


def _rates(lam, c):
    return -c * torch.nn.functional.softplus(lam.double())


def _gates(x, gl, lam, c):
    """alpha, i, n = sqrt(1 - alpha^2) and r in float64."""
    D = lam.numel()
    r, i = torch.sigmoid(gl[..., :D].double()), torch.sigmoid(gl[..., D:].double())
    log_a = _rates(lam, c) * r
    return torch.exp(log_a), i, torch.sqrt(-torch.expm1(2 * log_a)), r


def _exact_scan(case, seed):
    s = _scan_inputs(case, seed)
    B, L, D = case["B"], case["L"], case["D"]
    lam, c, gated = s["lam"].double(), case["c"], case["mode"] == "gated"
    real = torch.ones(B, L, 1, dtype=torch.bool, device="cuda")
    if s["lengths"] is not None:
        real = (torch.arange(L, device="cuda")[None] >= L - s["lengths"][:, None])[..., None]
    zero = torch.zeros(B, D, dtype=torch.float64, device="cuda")
    h0 = s["h0"].double() if s["h0"] is not None else zero
    a, i, n, r = _gates(s["x"], s["gl"], lam, c)
    x = s["x"].double()
    u = torch.where(real, n * i * x, 0.0)
    at = torch.where(real, a, 1.0).transpose(0, 1).contiguous()  # padding: the identity
    h = u.transpose(0, 1).contiguous()
    del u
    prev = h0
    for t in range(L):
        prev = h[t].addcmul_(at[t], prev)
    h_last = prev.clone()
    hb = h.transpose(0, 1)  # (B, L, D)
    sz = ds = None
    if gated:
        z = s["z"].double()
        sg = torch.sigmoid(z)
        sz, ds = z * sg, sg * (1 + z * (1 - sg))
        del z, sg
    y = hb * sz if gated else torch.where(real, hb, 0.0)
    out = {"y": y, "h_last": h_last}
    if not case["train"]:
        return out
    dy = torch.where(real, s["dh"].double(), 0.0)
    g = (dy * sz if gated else dy).transpose(0, 1).contiguous()
    w = s["dh_last"].double() if s["dh_last"] is not None else zero
    for t in range(L - 1, -1, -1):
        w = g[t].add_(w) * at[t]
    if case["state"]:
        out["dh0"] = w.clone()
    if gated:
        out["dz"] = dy * hb * ds
    del dy, sz, ds
    g = g.transpose(0, 1)
    hp = torch.empty(L, B, D, dtype=torch.float64, device="cuda")
    hp[0] = h0
    hp[1:] = h[:-1]
    del h, hb
    hp = hp.transpose(0, 1)
    dl = g * a * (hp - a * i * x / n)
    del hp
    out["dx"] = torch.where(real, g * n * i, 0.0)
    di = g * n * x * i * (1 - i)
    dr = dl * _rates(lam, c) * r * (1 - r)
    out["dgl"] = torch.where(real, torch.cat([dr, di], dim=2), 0.0)
    del di, dr
    out["dlam"] = -c * torch.sigmoid(lam) * torch.where(real, dl * r, 0.0).sum((0, 1))
    return out


def _exact_steps(case, seed):
    s = _step_inputs(case, seed)
    one = case["kind"] == "step"
    x, gl = (s["x"][:, None], s["gl"][:, None]) if one else (s["x"], s["gl"])
    a, i, n, _ = _gates(x, gl, s["lam"], case["c"])
    u = n * i * x.double()
    h, seq = s["h"].double(), []
    for k in range(x.shape[1]):
        h = a[:, k] * h + u[:, k]
        seq.append(h)
    return {"h": h} if one else {"h": h, "h_seq": torch.stack(seq, dim=1)}


def _exact_layer(case, seed):
    p, h, dy = _layer_inputs(case, seed)
    p = {k: v.double().requires_grad_() for k, v in p.items()}
    h, F = h.double().requires_grad_(), torch.nn.functional
    L, ed = case["L"], case["expand"] * case["d_model"]
    hx, hz = F.linear(h, p["in_proj.weight"], p["in_proj.bias"]).split(ed, dim=-1)
    xc = F.pad(hx.transpose(1, 2), (3, 0))
    conv = sum(xc[..., k:k + L] * p["conv.weight"][:, 0, k, None] for k in range(4))
    x = F.silu((conv + p["conv.bias"][:, None]).transpose(1, 2))
    gl = F.linear(x, p["gate_proj.weight"], p["gate_proj.bias"])
    a, i, n, _ = _gates(x, gl, p["lam"], 1.0)
    u, st, seq = n * i * x, 0.0, []
    for t in range(L):
        st = a[:, t] * st + u[:, t]
        seq.append(st)
    y = F.linear(torch.stack(seq, dim=1) * F.silu(hz), p["out_proj.weight"], p["out_proj.bias"])
    return (y, *torch.autograd.grad(y, [h, *(p[k] for k in LAYER_PARAMS)], dy.double()))


def exact(case, seed):
    kind = case["kind"]
    if kind == "layer":
        return tuple(t.detach() for t in _exact_layer(case, seed))
    return _exact_steps(case, seed) if kind in ("step", "steps") else _exact_scan(case, seed)
