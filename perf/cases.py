"""The work that a program hands to the LR-QAT library, as cases for timing.

Every case goes through the public binding (``paper_2406_06385_gb300.lrqat``) the way a
training loop, a range-setting script or a runtime calls it: buffers and workspaces are
allocated once, the calls are made on the current stream and nothing is synchronised.

Kinds of cases:
  step     one training step of a linear layer: forward and backward of each micro-batch
           (gradients accumulated over the micro-batches) and, with ``merge``, the fold into
           integer weights.  int8 activations per tensor are quantized once per step and both
           passes read their codes; per-token ones are quantized inside the calls.
  forward  the allocation-free forward of a runtime that owns all device memory.
  init     range setting of a layer before training: min-max and L^p scales and the downcast
           base of each.
  optim    the optimizer step on the adapters and scales of one decoder layer's projections:
           global gradient norm, then clipped AdamW on each projection.
"""
import math

import torch

from paper_2406_06385_gb300 import lrqat as LQ

DEV = "cuda"

# One layer and batch; a case names only what differs from these.
STEP = dict(kind="step", m=4096, k=4096, r=32, bits=4, group=0, phi=LQ.PHI_QFIXED, act=0, per_token=False, asym=False,
            u_bf16=False, T=8192, micro=1, merge=False)
FORWARD = dict(kind="forward", m=4096, k=4096, r=32, bits=4, group=0, phi=LQ.PHI_QFIXED, act=0, per_token=False,
               asym=False, u_bf16=False, T=16)
INIT = dict(kind="init", m=5120, k=5120, bits=4, group=0, phi=LQ.PHI_QFIXED, p_norm=2.0, candidates=100)
OPTIM = dict(kind="optim", d=5120, d_ff=13824, r=32, group=0)


def listed():
    return [
        # the smallest layer of the parity workloads: host work, launches and kernel start-up
        dict(STEP, name="tiny_step", m=256, k=256, r=4, T=64),
        # a serving runtime's call on a few tokens of a 7B attention projection
        dict(FORWARD, name="few_tokens_forward"),
        # gradient accumulation over two sequences of 1024 tokens (the paper's sequence length)
        dict(STEP, name="attn_2x1024", T=1024, micro=2),
        # a 7B attention projection on eight sequences of 1024 tokens
        dict(STEP, name="attn_8192"),
        # the INT2 runs: asymmetric grid, a batch with a ragged token count
        dict(STEP, name="attn_int2_2999", bits=2, asym=True, T=2999),
        # the weight-activation runs: dynamic int8 scale per token
        dict(STEP, name="attn_w4a8_4096", act=8, per_token=True, T=4096),
        # the largest rank of the paper's rank ablation
        dict(STEP, name="attn_r256", r=256),
        # a 7B gate/up projection, W3 on double-packed INT-3 storage
        dict(STEP, name="up_int3", m=11008, bits=3, phi=LQ.PHI_INT_PACKED),
        # an 8B down projection, group-wise W4 with static per-tensor int8 activations
        dict(STEP, name="down_g128_a8", k=14336, group=128, act=8),
        # a 13B gate projection on sixteen sequences, merged after the step: the largest
        dict(STEP, name="gate13b_16384", m=13824, k=5120, T=16384, merge=True),
        # range setting of a 13B attention projection with both estimators
        dict(INIT, name="init_5120"),
        # the optimizer step of one 13B decoder layer
        dict(OPTIM, name="optim_13b_layer"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _dim(rng, lo=256, hi=14336):
    """A layer dimension: the library takes multiples of 128, odd multiples among them."""
    return 128 * _log_int(rng, lo // 128, hi // 128)


def _quantizer(rng, c):
    """A weight quantizer of the paper's runs: bit width, storage, grid and granularity."""
    what = rng.choice(["q", "q", "int", "asym", "float", "u_bf16"])
    c["bits"] = rng.choice([2, 3, 4, 4])
    if what == "int":
        c["phi"] = LQ.PHI_INT_PACKED
    elif what == "asym":
        c.update(bits=2, asym=True)
    elif what == "float":
        c["phi"] = rng.choice([LQ.PHI_BF16, LQ.PHI_FP16, LQ.PHI_FP8_E4M3, LQ.PHI_FP8_E5M2])
    elif what == "u_bf16":
        c["u_bf16"] = True
    if rng.random() < 0.3:
        c["group"] = 128


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["forward"] * 2 + ["init", "optim"])
    if kind == "step":
        c = dict(STEP, m=_dim(rng), k=_dim(rng), r=rng.choice([4, 8, 16, 20, 32, 32, 64, 96, 128, 256]),
                 T=_log_int(rng, 48, 16384) | 1, merge=rng.random() < 0.2)
        if rng.random() < 0.3:
            c["T"] = max(64, c["T"] // 64 * 64)
        if rng.random() < 0.25:
            c.update(act=8, per_token=rng.random() < 0.5)
        _quantizer(rng, c)
        if c["r"] == 20:
            c["u_bf16"] = False
        while c["m"] * c["k"] * c["T"] > 13824 * 5120 * 16384:
            c["T"] = max(1, c["T"] // 2) | 1
        return c
    if kind == "forward":
        c = dict(FORWARD, m=_dim(rng, 512), k=_dim(rng, 512), r=rng.choice([8, 16, 20, 32, 64]), T=_log_int(rng, 1, 2048))
        _quantizer(rng, c)
        c["group"] = 0   # the fixed scratch holds the scale rows of small group-wise layers only
        if c["r"] == 20:
            c["u_bf16"] = False
        return c
    if kind == "init":
        return dict(INIT, m=_dim(rng, 512, 8192), k=_dim(rng, 512, 8192), bits=rng.choice([2, 3, 4]),
                    phi=rng.choice([LQ.PHI_QFIXED, LQ.PHI_INT_PACKED]), group=rng.choice([0, 0, 128]),
                    p_norm=rng.choice([2.0, 2.0, 2.4, 3.0, 3.5, 4.0, 5.0]), candidates=rng.choice([50, 80, 100]))
    return dict(OPTIM, d=_dim(rng, 1024, 5120), d_ff=_dim(rng, 2048, 14336), r=rng.choice([4, 16, 20, 32, 64, 128]),
                group=rng.choice([0, 0, 128]))


# ------------------------------------------------------------------------------ inputs

def _normal(g, shape, std, dtype=torch.float32):
    return torch.randn(shape, generator=g, device=DEV, dtype=torch.float32).mul_(std).to(dtype)


def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _weights(c, g):
    """Pretrained weights: N(0, 0.02) with 0.1% outliers ten times as large; with the asymmetric
    grid every row is shifted, so that the zero offsets spread over the grid."""
    W0 = _normal(g, (c["m"], c["k"]), 0.02)
    out = torch.rand(W0.shape, generator=g, device=DEV) < 1e-3
    W0 = torch.where(out, W0 * 10, W0)
    if c.get("asym"):
        W0 += (torch.rand((c["m"], 1), generator=g, device=DEV) * 2 - 1) * 0.03
    return W0


def _adapters(c, g):
    """Adapters in mid-training: B is no longer zero, so A B moves codes."""
    A = _normal(g, (c["m"], c["r"]), 1 / 64, torch.bfloat16)
    B = _normal(g, (c["r"], c["k"]), 1e-3, torch.bfloat16)
    return A, B


def _batch(c, g):
    X = _normal(g, (c["T"], c["k"]), 1.0, torch.bfloat16)
    dY = _normal(g, (c["T"], c["m"]), 1.0, torch.bfloat16) if c["kind"] == "step" else None
    return X, dY


def _s_x(X):
    """A static activation scale set on calibration data: a few values of a batch clip."""
    return (X.float().abs().amax() / 127.0 * 0.9).reshape(1)


def _scale_shape(c):
    return (c["m"], c["k"] // c["group"]) if c["group"] else (c["m"],)


def _layer(c, r, zero=None):
    return LQ.Layer(c["m"], c["k"], r, float(r), c["bits"], c["group"], c["phi"], c.get("act", 0),
                    None if zero is None else zero.data_ptr(), int(c.get("per_token", False)),
                    int(c.get("u_bf16", False)))


def _base_buffer(c):
    if c["phi"] == LQ.PHI_INT_PACKED:
        return torch.empty((c["m"], c["k"] // 2), dtype=torch.uint8, device=DEV)
    dtype = {LQ.PHI_QFIXED: torch.int8, LQ.PHI_BF16: torch.int16, LQ.PHI_FP16: torch.int16}.get(c["phi"], torch.uint8)
    return torch.empty((c["m"], c["k"]), dtype=dtype, device=DEV)


def _empty(shape, dtype):
    return torch.empty(shape, dtype=dtype, device=DEV)


# ----------------------------------------------------------------------------- prepare

def prepare(case, seed):
    return {"step": _prepare_layer, "forward": _prepare_layer, "init": _prepare_init,
            "optim": _prepare_optim}[case["kind"]](case, _generator(seed))


def _prepare_layer(c, g):
    W0 = _weights(c, g)
    A, B = _adapters(c, g)
    s = _empty(_scale_shape(c), torch.float32)
    z = torch.empty_like(s) if c["asym"] else None
    L = _layer(c, c["r"], z)
    phi0 = _base_buffer(c)
    LQ.range_minmax(L, W0, s)
    LQ.downcast(L, W0, s, phi0)
    batches = [_batch(c, g) for _ in range(c.get("micro", 1))]
    static = c["act"] == 8 and not c["per_token"]
    st = dict(c=c, L=L, z=z, phi0=phi0, s=s, A=A, B=B, batches=batches, s_x=_s_x(batches[0][0]) if static else None)
    T, m, k, r = c["T"], c["m"], c["k"], c["r"]
    st["Y"] = [_empty((T, m), torch.bfloat16) for _ in batches]
    if c["kind"] == "forward":
        return st
    st["dX"] = [_empty((T, k), torch.bfloat16) for _ in batches]
    st["dA"], st["dB"], st["ds"] = _empty((m, r), torch.float32), _empty((r, k), torch.float32), torch.empty_like(s)
    st["ws_f"] = _empty(max(LQ.fwd_workspace_bytes(L, T), 16), torch.uint8)
    st["ws_b"] = _empty(LQ.bwd_workspace_bytes(L, T), torch.uint8)
    if static:
        st["X_q"], st["mask"] = _empty((T, k), torch.bfloat16), _empty((k, (T + 31) // 32), torch.int32)
    if c["merge"]:
        st["W_Z"] = _empty((m, k), torch.int8)
    return st


def _prepare_init(c, g):
    n = _scale_shape(c)
    return dict(c=c, L=_layer(c, 1), W0=_weights(c, g), s_mm=_empty(n, torch.float32), s_lp=_empty(n, torch.float32),
                phi_mm=_base_buffer(c), phi_lp=_base_buffer(c))


def _projections(c):
    d, f = c["d"], c["d_ff"]
    return [(d, d)] * 4 + [(f, d), (f, d), (d, f)]


ADAM = dict(lr_ab=1e-3, lr_s=1e-5, beta1=0.9, beta2=0.95, eps=1e-8, step=100, max_grad_norm=1.0)


def _optim_sizes(c):
    """Elements of A, B and s of each projection."""
    return [(m * c["r"], c["r"] * k, m * (k // c["group"] if c["group"] else 1)) for m, k in _projections(c)]


def _optim_flat(c, g):
    """Parameters, gradients and optimizer state of a decoder layer, each kind in one flat buffer."""
    nA, nB, ns = (sum(n) for n in zip(*_optim_sizes(c)))
    flat = dict(dA=_normal(g, (nA,), 1e-2), dB=_normal(g, (nB,), 1e-2), ds=_normal(g, (ns,), 1e-2),
                A32=_normal(g, (nA,), 1 / 64), B32=_normal(g, (nB,), 1e-3),
                s=_normal(g, (ns,), 1e-3).abs_().add_(1e-2),
                mA=_normal(g, (nA,), 1e-5), mB=_normal(g, (nB,), 1e-5), ms=_normal(g, (ns,), 1e-5),
                vA=_normal(g, (nA,), 1e-5).square_(), vB=_normal(g, (nB,), 1e-5).square_(),
                vs=_normal(g, (ns,), 1e-5).square_())
    flat["A"], flat["B"] = flat["A32"].to(torch.bfloat16), flat["B32"].to(torch.bfloat16)
    return flat


def _prepare_optim(c, g):
    """The projections' tensors are views of the flat buffers."""
    flat = _optim_flat(c, g)
    layers, oa, ob, os = [], 0, 0, 0
    for (m, k), (na, nb, n) in zip(_projections(c), _optim_sizes(c)):
        at = {key: flat[key][oa:oa + na] for key in ("dA", "A32", "mA", "vA", "A")}
        at.update({key: flat[key][ob:ob + nb] for key in ("dB", "B32", "mB", "vB", "B")})
        at.update({key: flat[key][os:os + n] for key in ("ds", "s", "ms", "vs")})
        layers.append((LQ.Layer(m, k, c["r"], float(c["r"]), 4, c["group"], LQ.PHI_QFIXED, 0), at))
        oa, ob, os = oa + na, ob + nb, os + n
    return dict(c=c, flat=flat, layers=layers, sqnorm=torch.zeros(1, dtype=torch.float32, device=DEV),
                opt=LQ.AdamW.make(ADAM["lr_ab"], ADAM["lr_s"], ADAM["step"], ADAM["beta1"], ADAM["beta2"], ADAM["eps"],
                                  max_grad_norm=ADAM["max_grad_norm"]))


# --------------------------------------------------------------------------------- run

def run(state):
    return {"step": _run_step, "forward": _run_forward, "init": _run_init, "optim": _run_optim}[state["c"]["kind"]](state)


def _run_step(st):
    c, L, T = st["c"], st["L"], st["c"]["T"]
    par = (st["phi0"], st["s"], st["A"], st["B"], st["s_x"])
    for i, ((X, dY), Y, dX) in enumerate(zip(st["batches"], st["Y"], st["dX"])):
        if "X_q" in st:
            LQ.act_quant(L, T, X, st["s_x"], st["X_q"], st["mask"])
            LQ.linear_fwd_quantized(L, T, st["X_q"], *par, Y, st["ws_f"])
            LQ.linear_bwd_quantized(L, T, dY, st["X_q"], st["mask"], *par, dX, st["dA"], st["dB"], st["ds"], i > 0,
                                    st["ws_b"])
        else:
            LQ.linear_fwd(L, T, X, *par, Y, st["ws_f"])
            LQ.linear_bwd(L, T, dY, X, *par, dX, st["dA"], st["dB"], st["ds"], i > 0, st["ws_b"])
    out = dict(Y=st["Y"], dX=st["dX"], dA=st["dA"], dB=st["dB"], ds=st["ds"])
    if c["merge"]:
        LQ.merge(L, st["phi0"], st["A"], st["B"], st["W_Z"])
        out["W_Z"] = st["W_Z"]
    return out


def _run_forward(st):
    LQ.linear_fwd_noalloc(st["L"], st["c"]["T"], st["batches"][0][0], st["phi0"], st["s"], st["A"], st["B"], st["s_x"],
                          st["Y"][0])
    return dict(Y=st["Y"])


def _run_init(st):
    c, L, W0 = st["c"], st["L"], st["W0"]
    LQ.range_minmax(L, W0, st["s_mm"])
    LQ.downcast(L, W0, st["s_mm"], st["phi_mm"])
    LQ.range_lp(L, W0, st["s_lp"], c["p_norm"], c["candidates"])
    LQ.downcast(L, W0, st["s_lp"], st["phi_lp"])
    return {n: st[n] for n in ("s_mm", "phi_mm", "s_lp", "phi_lp")}


OPTIM_OUT = ("A32", "B32", "s", "mA", "vA", "mB", "vB", "ms", "vs", "A", "B")


def _run_optim(st):
    st["sqnorm"].zero_()
    for L, t in st["layers"]:
        LQ.grad_sqnorm(L, t["dA"], t["dB"], t["ds"], st["sqnorm"])
    for L, t in st["layers"]:
        LQ.adamw_step(L, st["opt"], st["sqnorm"], t["dA"], t["dB"], t["ds"], t, t["s"], t["A"], t["B"])
    return {n: st["flat"][n] for n in OPTIM_OUT} | dict(sqnorm=st["sqnorm"])


# -------------------------------------------------------------------------------- work

def _base_bytes(c):
    per = {LQ.PHI_INT_PACKED: 0.5, LQ.PHI_BF16: 2.0, LQ.PHI_FP16: 2.0}.get(c["phi"], 1.0)
    return per * c["m"] * c["k"]


def work(case):
    c = case
    if c["kind"] == "optim":
        n = sum(c["r"] * (m + k) for m, k in _projections(c))
        ns = sum(m * (k // c["group"] if c["group"] else 1) for m, k in _projections(c))
        # gradient, parameter and two moments in; parameter, moments and the bf16 copy out
        return {"bytes": 30.0 * n + 28.0 * ns, "flops": 14.0 * (n + ns)}
    m, k = c["m"], c["k"]
    ns = m * (k // c["group"] if c["group"] else 1)
    if c["kind"] == "init":
        # the weights in, two scales and two bases out; per weight and candidate a scaled
        # rounding, two clip bounds, the error and its power
        return {"bytes": 4.0 * m * k + 8.0 * ns + 2 * _base_bytes(c), "flops": 7.0 * m * k * c["candidates"]}
    T, r = c["T"], c["r"]
    par = _base_bytes(c) + 4.0 * ns * (2 if c["asym"] else 1) + 2.0 * r * (m + k)
    if c["kind"] == "forward":
        return {"bytes": 2.0 * T * (m + k) + par, "flops": 2.0 * T * m * k + 2.0 * r * m * k}
    n = c["micro"]
    grads = 4.0 * (r * (m + k) + ns)
    return {"bytes": n * 4.0 * T * (m + k) + par + grads + (1.0 * m * k if c["merge"] else 0.0),
            "flops": n * (6.0 * T * m * k + 4.0 * r * m * k) + 2.0 * r * m * k}


# ------------------------------------------------------------------- values in 64 bits

def exact(case, seed):
    return {"step": _exact_layer, "forward": _exact_layer, "init": _exact_init,
            "optim": _exact_optim}[case["kind"]](case, _generator(seed))


def _div32(a, b):
    """The fp32 quotient of fp32 values, in 64 bits: rounding the 64-bit quotient gives it."""
    return (a.double() / b.double()).float().double()


def _grid(c):
    return -float(2 ** (c["bits"] - 1)), float(2 ** (c["bits"] - 1) - 1)


def _segments(c, t):
    """[m, k] as [m, groups, group width] (one group per row per channel)."""
    return t.reshape(c["m"], -1, c["group"] or c["k"])


def _range(c, W0):
    n, p = _grid(c)
    w = _segments(c, W0).double()
    if not c.get("asym"):
        a = w.abs().amax(-1)
        return torch.where(a > 0, a / p, torch.ones_like(a)).float().double(), None
    lo, hi = w.amin(-1), w.amax(-1)
    span = (hi - lo).float().double()
    s = torch.where(span > 0, span / (2 ** c["bits"] - 1), torch.ones_like(span)).float().double()
    return s, torch.clamp(torch.round(n - _div32(lo, s)), n, p)


def _base(c, W0, s, z):
    """phi^{-1}(phi(W0 / s)) as 64-bit values."""
    n, p = _grid(c)
    q = _div32(_segments(c, W0), s.unsqueeze(-1))
    if z is not None:
        q = q + z.unsqueeze(-1)
    if c["phi"] == LQ.PHI_QFIXED:
        f = float(2 ** (8 - c["bits"]))
        q = torch.round(q.clamp(n, p) * f) / f
    elif c["phi"] == LQ.PHI_INT_PACKED:
        q = torch.round(q).clamp(n, p)
    else:
        dtype, top = {LQ.PHI_BF16: (torch.bfloat16, None), LQ.PHI_FP16: (torch.float16, 65504.0),
                      LQ.PHI_FP8_E4M3: (torch.float8_e4m3fn, 448.0), LQ.PHI_FP8_E5M2: (torch.float8_e5m2, 57344.0)}[c["phi"]]
        q = q if top is None else q.clamp(-top, top)
        q = q.float().to(dtype).double()
    return q.reshape(c["m"], c["k"])


def _spread(c, t):
    """A scale or offset per row or group -> one per weight (broadcast along a row per channel)."""
    return t.repeat_interleave(c["group"], 1) if c["group"] else t


def _exact_layer(c, g):
    if c["m"] * c["k"] * c["T"] * c.get("micro", 1) > 13824 * 5120 * 16384:
        return None
    W0 = _weights(c, g)
    A, B = (t.double() for t in _adapters(c, g))
    n, p = _grid(c)
    s, z = _range(c, W0)
    base = _base(c, W0, s, z)
    del W0
    if c["u_bf16"]:
        u = (base + (A @ B).to(torch.bfloat16).double()).to(torch.bfloat16).double()
    else:
        u = base + A @ B
    del base
    w = torch.round(u)
    M = (w >= n) & (w <= p)
    w = w.clamp(n, p)
    del u
    if z is not None:
        w = w - _spread(c, z)
    sw = _spread(c, s)
    out, G = dict(Y=[], dX=[]), 0
    s_x = None
    for i in range(c.get("micro", 1)):
        X, dY = _batch(c, g)
        X, mask = X.double(), None
        if c["act"] == 8:
            if c["per_token"]:
                a = X.abs().amax(-1, keepdim=True)
                sx = torch.where(a > 0, a / 127, torch.ones_like(a)).float().double()
            else:
                s_x = _s_x(X.to(torch.bfloat16)).double() if s_x is None else s_x
                sx = s_x
            q = torch.round(_div32(X, sx))
            mask = None if c["per_token"] else (q >= -128) & (q <= 127)
            X = sx * q.clamp(-128, 127)
        out["Y"].append(X @ (w * sw).t())
        if c["kind"] == "forward":
            continue
        dX = dY.double() @ (w * sw)
        out["dX"].append(dX if mask is None else dX * mask)
        G = G + dY.double().t() @ X
        del X, dY, dX
    if c["kind"] == "forward":
        return dict(Y=out["Y"])
    out["ds"] = _segments(c, G * w).sum(-1).reshape(_scale_shape(c))
    dU = G.mul_(sw).mul_(M)
    out["dA"], out["dB"] = dU @ B.t(), A.t() @ dU
    if c["merge"]:
        out["W_Z"] = None   # whole numbers
    return out


def _exact_init(c, g):
    W0 = _weights(c, g)
    n, p = _grid(c)
    s_mm, _ = _range(c, W0)
    w = _segments(c, W0).double()
    best = torch.full(s_mm.shape, float("inf"), device=DEV, dtype=torch.float64)
    s_lp = torch.zeros_like(s_mm)
    for j in range(1, c["candidates"] + 1):
        s = (s_mm * j / c["candidates"]).float().double()
        e = torch.round(_div32(w, s.unsqueeze(-1))).clamp_(n, p).mul_(s.unsqueeze(-1)).sub_(w).abs_()
        loss = e.pow_(c["p_norm"]).sum(-1)
        better = loss < best
        best, s_lp = torch.where(better, loss, best), torch.where(better, s, s_lp)
    shape = _scale_shape(c)
    return dict(s_mm=s_mm.reshape(shape), phi_mm=None, s_lp=s_lp.reshape(shape), phi_lp=None)


def _exact_optim(c, g):
    f = {n: t.double() for n, t in _optim_flat(c, g).items()}
    sq = sum(f[n].square().sum() for n in ("dA", "dB", "ds"))
    coef = torch.clamp(ADAM["max_grad_norm"] / (sq.sqrt() + 1e-6), max=1.0)
    f32 = lambda v: float(torch.tensor(v, dtype=torch.float32))   # the hyperparameters as the call takes them
    b1, b2, eps = f32(ADAM["beta1"]), f32(ADAM["beta2"]), f32(ADAM["eps"])
    out = {}
    for par, grad, m, v, lr in (("A32", "dA", "mA", "vA", f32(ADAM["lr_ab"])), ("B32", "dB", "mB", "vB", f32(ADAM["lr_ab"])),
                                ("s", "ds", "ms", "vs", f32(ADAM["lr_s"]))):
        gr = coef * f[grad]
        out[m] = b1 * f[m] + (1 - b1) * gr
        out[v] = b2 * f[v] + (1 - b2) * gr * gr
        mh, vh = out[m] / (1 - b1 ** ADAM["step"]), out[v] / (1 - b2 ** ADAM["step"])
        out[par] = f[par] - lr * mh / (vh.sqrt() + eps)
    out["A"], out["B"] = out["A32"].clone(), out["B32"].clone()
    return {n: out[n] for n in OPTIM_OUT} | dict(sqnorm=sq.reshape(1))

