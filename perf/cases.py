"""What this framework is timed on: passes through its public entry points.

Each case is one pass of a kind of work that a program using the library does
over and over, at sizes from the library's own workloads and tests:

* "step"     two optimisation steps of the quantizer on one weight matrix
             (forward and backward each; under the local mapping the first
             remaps the codes and the second keeps them);
* "fused"    two fused optimisation steps (backward, SGD update, next
             forward; the second remaps);
* "omni", "awq"  two forwards (remap, keep) and a backward with OmniQuant's
             and AWQ's transformations;
* "init"     the unified initialization of a matrix;
* "export"   Theorem 1 and the bit-planes of a matrix;
* "product"  the deployment product of the exported format with some tokens.
"""

import math

import torch

from paper_2506_03781_gb300 import api

LR_F, LR_B = 0.005, 0.0005
INIT_G, INIT_T = 30, 15
PARAMS = ("delta", "zu", "s", "sr", "alpha", "zb")
WIDTH = {"bf16": 2, "f32": 4}
CHUNK = 1 << 22                      # elements that exact() works on at a time


def _case(name, kind, out, n_in, q=3, g=128, dtype="bf16", **more):
    return dict(name=name, kind=kind, out=out, n_in=n_in, q=q, g=g, dtype=dtype, **more)


def listed():
    return [
        # the smallest matrix of the workloads, fp32: launches and host calls count
        _case("step_small_f32", "step", 1024, 1024, dtype="f32", map="local", filter="ste"),
        # the MLP matrix of the benchmark
        _case("step_mlp", "step", 14336, 4096, map="local", filter="ste"),
        # rows that are no whole number of 512-column units: 86 groups of 128, full mapping
        _case("step_ragged_full", "step", 4096, 11008, q=4, map="full", filter="ste"),
        # an attention projection in larger groups than the usual ones, the whole-element filter
        _case("step_attn_g256", "step", 4096, 4096, q=2, g=256, map="local", filter="element"),
        # the fused step on a down projection (long rows), bf16 gradients and outputs
        _case("fused_down_bf16", "fused", 4096, 14336, q=2, g=64, io="bf16"),
        # the other two transformations, on the MLP matrix
        _case("omni_mlp", "omni", 14336, 4096),
        _case("awq_mlp", "awq", 14336, 4096),
        # before training: a key/value projection initialised with the paper's grid and rounds
        _case("init_kv", "init", 1024, 4096),
        # after training: the MLP matrix in the deployment format
        _case("export_mlp", "export", 14336, 4096, mode="reuse", half=False),
        # deployment: one token against the MLP matrix (decode)
        _case("product_1", "product", 14336, 4096, batch=1),
        # a prefill chunk or a batch of requests against the same matrix
        _case("product_64", "product", 14336, 4096, batch=64),
        # a small batch of fp32 activations against the largest down projection
        _case("product_70b_f32", "product", 8192, 28672, dtype="f32", batch=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Kinds as listed; matrices of 64 to 14336 rows (any number) by 512 to
    14336 columns (a multiple of the group), group sizes and bit-widths as the
    library takes them."""
    kind = rng.choice(["step", "step", "step", "fused", "omni", "awq", "init", "export", "product", "product"])
    q = rng.choice([2, 2, 3, 3, 3, 4, 4, 1])
    g = rng.choice([32, 64, 64, 128, 128, 128, 256, 512])
    if kind == "fused":
        g = min(g, 128)
    out = _log(rng, 64, 14336)
    n_in = max(1, _log(rng, 512, 14336) // g) * g
    c = dict(kind=kind, out=out, n_in=n_in, q=q, g=g, dtype=rng.choice(["bf16", "bf16", "f32"]))
    if kind == "step":
        c.update(map=rng.choice(["local", "local", "full"]), filter=rng.choice(["ste", "ste", "ste", "element"]))
    elif kind == "fused":
        c.update(n_in=max(512, n_in // 512 * 512), io=rng.choice(["bf16", "f32"]))
    elif kind == "init":
        n_in = min(n_in, 4096)
        most = 2 ** 25 // (n_in << q) if g <= 128 else 128
        c.update(n_in=n_in, out=_log(rng, 32, max(32, min(1024, most))))
    elif kind == "export":
        c.update(mode=rng.choice(["reuse", "reuse", "eq4"]), half=rng.choice([False, True]))
    elif kind == "product":
        c.update(batch=_log(rng, 1, 64))
    big = 14336 * 4096
    if c["out"] * c["n_in"] > big:
        c["out"] = max(64, big // c["n_in"])
    return c


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _randn(gen, *shape):
    return torch.randn(*shape, generator=gen, device="cuda")


def _weights(gen, out, n_in, dtype):
    """Student-t(4) weights of standard deviation 0.02, one column in a thousand ten times larger."""
    w = _randn(gen, out, n_in)
    v = torch.zeros_like(w)
    for _ in range(4):
        v += _randn(gen, out, n_in).square_()
    w = w.div_(v.mul_(0.25).sqrt_()).mul_(0.02 / math.sqrt(2.0))
    cols = torch.randperm(n_in, generator=gen, device="cuda")[:max(1, n_in // 1000)]
    w[:, cols] *= 10.0
    return w.to(torch.bfloat16) if dtype == "bf16" else w


def _spread(gen, t, eps):
    return t * (1.0 + eps * _randn(gen, *t.shape))


def _groups(t, g):
    return t.reshape(t.shape[0], t.shape[1] // g, g)


def _clip_params(gen, wg, q, eps):
    """Delta, zero point, alpha, z_B of clipped uniform levels, each but the zero points spread by eps."""
    top = 2 ** q - 1
    lo, hi = wg.amin(-1).float(), wg.amax(-1).float()
    delta = 0.8 * (hi - lo) / top
    zero = -0.8 * lo / delta
    alpha = 0.5 * 2.0 ** torch.arange(q, device="cuda").expand(*delta.shape, q)
    return _spread(gen, delta, eps), zero, _spread(gen, alpha, eps).contiguous(), torch.full_like(delta, top / 2)


def _codes(wg, delta, zero, q, shape):
    """With uniform levels the code word is the rounded, clamped weight."""
    x = wg.float() / delta[..., None] + zero[..., None]
    return x.round_().clamp_(0, 2 ** q - 1).to(torch.uint8).reshape(shape)


def _flexround(gen, W, q, g, eps=0.01):
    out, n_in = W.shape
    wg = _groups(W, g)
    delta, zu, alpha, zb = _clip_params(gen, wg, q, eps)
    p = {"delta": delta, "zu": zu, "s": 1.0 + eps * _randn(gen, out, n_in), "sr": 1.0 + eps * _randn(gen, out),
         "alpha": alpha, "zb": zb}
    return p, _codes(wg, delta, zu, q, (out, n_in))


def prepare(case, seed):
    kind, out, n_in, q, g = (case[k] for k in ("kind", "out", "n_in", "q", "g"))
    gen = _gen(seed)
    s = {"case": case}
    if kind == "product":
        s["planes"] = torch.randint(-2 ** 31, 2 ** 31, (q, out, n_in // 32), generator=gen, device="cuda",
                                    dtype=torch.int32)
        step = 0.02 * (1.0 + 0.2 * _randn(gen, out, n_in // g))
        s["alpha"] = _spread(gen, 0.5 * step[..., None] * 2.0 ** torch.arange(q, device="cuda"), 0.05).contiguous()
        s["zb"] = 0.1 * step * _randn(gen, out, n_in // g)
        x = _randn(gen, case["batch"], n_in)
        s["x"] = x.to(torch.bfloat16) if case["dtype"] == "bf16" else x
        s["y"] = torch.empty(case["batch"], out, device="cuda")
        s["work"] = api.bcq_gemv_workspace(out, n_in, case["batch"])
        return s
    W = s["W"] = _weights(gen, out, n_in, case["dtype"])
    if kind == "init":
        s["params"] = api.empty_params(out, n_in, q, g)
        s["codes"] = torch.empty(out, n_in, dtype=torch.uint8, device="cuda")
        return s
    grad = 0.01 * _randn(gen, out, n_in)
    if kind == "step":
        # the parameters of two successive steps: the second set is the first
        # moved by about what an SGD step moves it
        p0, s["codes"] = _flexround(gen, W, q, g)
        p1 = {k: (_spread(gen, v, 3e-4) if k in ("delta", "s", "sr", "alpha") else v.clone()) for k, v in p0.items()}
        s["grad"], s["steps"] = grad, []
        for p in (p0, p1):
            what, grads = torch.empty(out, n_in, device="cuda"), api.empty_grads(out, n_in, q, g)
            s["steps"].append((api.Quantizer(W, q, g, p, s["codes"], what, grad, grads), p, what, grads))
    elif kind == "fused":
        s["params"], s["codes"] = _flexround(gen, W, q, g)
        io = torch.bfloat16 if case["io"] == "bf16" else torch.float32
        s["grad"] = (1e-4 * grad).to(io)
        s["what"] = [torch.empty(out, n_in, dtype=io, device="cuda") for _ in range(2)]
    elif kind == "omni":
        Gr = n_in // g
        _, _, alpha, zb = _clip_params(gen, _groups(W, g), q, 0.01)
        s["params"] = {"beta": 0.8 * (1.0 + 0.02 * _randn(gen, out, Gr)), "gamma": 0.8 * (1.0 + 0.02 * _randn(gen, out, Gr)),
                       "alpha": alpha, "zb": zb}
        delta, zo = _omni_scales(_groups(W, g).float(), s["params"], q)
        s["codes"] = _codes(_groups(W, g), delta, zo, q, (out, n_in))
        s["grads"] = {"d" + k: torch.empty_like(v) for k, v in s["params"].items()}
    elif kind == "awq":
        sa = torch.exp(0.2 * _randn(gen, n_in))
        scaled = _groups(W.float() * sa, g)
        delta, za, alpha, zb = _clip_params(gen, scaled, q, 0.01)
        s["params"] = {"sa": sa, "delta": delta, "za": za, "alpha": alpha, "zb": zb}
        s["codes"] = _codes(scaled, delta, za, q, (out, n_in))
        s["grads"] = {"d" + k: torch.empty_like(v) for k, v in s["params"].items()}
        s["work"] = torch.empty(max(4, api.uq_awq_bwd_workspace_bytes(out, n_in, q, g) // 4), device="cuda")
    elif kind == "export":
        s["params"], s["codes"] = _flexround(gen, W, q, g)
        real = torch.float16 if case["half"] else torch.float32
        s["planes"] = torch.empty(q, out, n_in // 32, dtype=torch.int32, device="cuda")
        s["alpha"] = torch.empty(out, n_in // g, q, dtype=real, device="cuda")
        s["zb"] = torch.empty(out, n_in // g, dtype=real, device="cuda")
    if kind in ("omni", "awq"):
        s["grad"] = grad
        s["what"] = [torch.empty(out, n_in, device="cuda") for _ in range(2)]
    return s


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------

def run(s):
    case = s["case"]
    kind, q, g = case["kind"], case["q"], case["g"]
    if kind == "step":
        mode = api.MAP_FULL if case["map"] == "full" else api.MAP_LOCAL_PERIODIC
        res = {"codes": s["codes"]}
        for i, (qz, p, what, grads) in enumerate(s["steps"]):
            qz.fwd(i, 2, mode)
            if case["filter"] == "element":
                api.uq_quantize_bwd_ex(s["W"], q, g, p, s["codes"], s["grad"], grads, api.FILTER_ELEMENT)
            else:
                qz.bwd()
            res["what%d" % i], res["grads%d" % i] = what, grads
        return res
    if kind == "fused":
        call = api.uq_train_step_bf16 if case["io"] == "bf16" else api.uq_train_step
        for i in range(2):
            call(s["W"], q, g, s["params"], s["codes"], s["grad"], s["what"][i], i, LR_F, LR_B)
        return {"codes": s["codes"], "params": s["params"], "what0": s["what"][0], "what1": s["what"][1]}
    if kind in ("omni", "awq"):
        fwd, bwd = ((api.uq_quantize_fwd_omni, api.uq_quantize_bwd_omni) if kind == "omni" else
                    (api.uq_quantize_fwd_awq, api.uq_quantize_bwd_awq))
        for i in range(2):
            fwd(s["W"], q, g, s["params"], s["codes"], s["what"][i], step=i)
        more = {} if kind == "omni" else {"workspace": s["work"]}
        bwd(s["W"], q, g, s["params"], s["codes"], s["grad"], s["grads"], **more)
        return {"codes": s["codes"], "grads": s["grads"], "what0": s["what"][0], "what1": s["what"][1]}
    if kind == "init":
        api.uq_init_params(s["W"], q, g, s["params"], s["codes"], G=INIT_G, T=INIT_T)
        return {"codes": s["codes"], "params": s["params"]}
    if kind == "export":
        call = api.uq_export_bcq_half if case["half"] else api.uq_export_bcq
        call(s["W"], q, g, s["params"], s["codes"], s["planes"], s["alpha"], s["zb"],
             api.EXPORT_REUSE_CODES if case["mode"] == "reuse" else api.EXPORT_REMAP_EQ4)
        return {"alpha": s["alpha"], "planes": s["planes"], "zb": s["zb"]}
    api.uq_bcq_gemv(s["planes"], s["alpha"], s["zb"], s["x"], s["y"], g, workspace=s["work"])
    return s["y"]


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------

def work(case):
    kind, out, n_in, q, g = (case[k] for k in ("kind", "out", "n_in", "q", "g"))
    n, w = out * n_in, WIDTH[case["dtype"]]
    gp = 4 * (n // g) * (3 + q)                        # the group parameters
    L = 2 ** q
    if kind == "step":
        bwd = n * (w + 4 + 1 + 4 + 4) + 2 * gp + 8 * out
        full = n * (w + 4 + 4 + 1) + gp + 4 * out
        if case["map"] == "full":
            return {"bytes": 2 * (full + bwd), "flops": n * 2 * (3 + 2 * L + 2 + 12 + q)}
        remap, keep = full + n, n * (1 + 4) + gp
        return {"bytes": remap + keep + 2 * bwd, "flops": n * (3 + 6 + 2 + 2 + 2 * (12 + q))}
    if kind == "fused":
        io = WIDTH[case["io"]]
        each = n * (w + 4 + 1 + io + 4 + io) + 2 * gp + 8 * out
        return {"bytes": 2 * each + n, "flops": n * 2 * (22 + q)}
    if kind == "omni":
        return {"bytes": n * ((w + 1 + 4 + 1) + (w + 1 + 4) + (w + 1 + 4)) + 4 * gp, "flops": n * (30 + q)}
    if kind == "awq":
        return {"bytes": n * ((w + 1 + 4 + 1) + (1 + 4) + (w + 1 + 4)) + 4 * gp + 16 * n_in, "flops": n * (30 + q)}
    if kind == "init":
        # every candidate: the transformation, the greedy start, two rounds of
        # the nearest level and the error (a fixed point ends the rounds early)
        return {"bytes": n * (w + 4 + 1) + gp + 4 * out, "flops": n * INIT_G * (3 + q * (q + 1) + 2 * 2 * L + 2 * L + 4)}
    if kind == "export":
        real = 2 if case["half"] else 4
        src = n if case["mode"] == "reuse" else n * w
        return {"bytes": src + q * n // 8 + gp + real * (n // g) * (q + 1),
                "flops": 0 if case["mode"] == "reuse" else n * 2 * L}
    b = case["batch"]
    return {"bytes": q * n // 8 + 4 * (n // g) * (q + 1) + b * n_in * w + 4 * b * out, "flops": 2 * n * b}


def tolerance(case):
    kind = case["kind"]
    if kind == "export":
        return "exact"                                 # one rounding per value, whole words otherwise
    if kind == "fused":
        # a parameter rounded the other way moves a code that lies on the
        # border of two levels: about one in ten million
        return {"rel": 5e-4, "max": 0.999, "differ": 1e-6}
    if kind == "init":
        return {"rel": 1e-5, "max": 1e-2, "differ": 1e-5}    # alpha of a group or two rounds the other way
    return {"rel": 1e-5}                               # fp32 sums that cancel: 1e-7 to 1e-6 from their 64-bit values


# --------------------------------------------------------------------------
# 64-bit results
# --------------------------------------------------------------------------
#
# Decisions (codes, the filter) are whole numbers, taken in fp32 in the order
# that the entry points state; every value that follows from them is in 64 bits.

def _signs(q):
    c = torch.arange(2 ** q, device="cuda")
    return torch.stack([((c >> j) & 1) * 2 - 1 for j in range(q)]).to(torch.float64)      # [q, L]


def _levels32(alpha, zb):
    """fp32 levels by code word, added in the stated order."""
    s = _signs(alpha.shape[-1]).float()
    lv = s[0] * alpha[..., :1]
    for j in range(1, alpha.shape[-1]):
        lv = lv + s[j] * alpha[..., j:j + 1]
    return lv + zb[..., None]


def _nearest(x, lv):
    srt, order = torch.sort(lv, dim=-1, stable=True)
    best = (x - srt[..., :1]).abs()
    rank = torch.zeros_like(x, dtype=torch.int64)
    for r in range(1, lv.shape[-1]):
        d = (x - srt[..., r:r + 1]).abs()
        rank = torch.where(d < best, r, rank)
        best = torch.minimum(best, d)
    return torch.gather(order, -1, rank)


def _remap(x, lv, codes):
    srt, order = torch.sort(lv, dim=-1, stable=True)
    rank = torch.argsort(order, dim=-1)
    d = torch.gather(rank, -1, codes)
    best, new = (x - torch.gather(srt, -1, d)).abs(), d
    for near in ((d - 1).clamp_min(0), (d + 1).clamp_max(lv.shape[-1] - 1)):
        dist = (x - torch.gather(srt, -1, near)).abs()
        new = torch.where(dist < best, near, new)
        best = torch.minimum(best, dist)
    return torch.gather(order, -1, new)


def _map(x, alpha, zb, codes, mode):
    if mode == "keep":
        return codes
    lv = _levels32(alpha.float(), zb.float())
    return _nearest(x, lv) if mode == "full" else _remap(x, lv, codes)


def _value(alpha, zb, codes):
    """l(code) in the type of the parameters."""
    lv = (alpha[..., None] * _signs(alpha.shape[-1]).to(alpha.dtype)).sum(-2) + zb[..., None]
    return torch.gather(lv, -1, codes)


def _filter(x32, alpha, zb, codes):
    m = torch.gather(_levels32(alpha.float(), zb.float()), -1, codes)
    return ((x32 - m).abs() <= alpha.float().abs().amin(-1, keepdim=True)).double()


def _dalpha(G, codes, q):
    return torch.stack([(G * (((codes >> j) & 1) * 2 - 1)).sum(-1) for j in range(q)], -1)


def _x32(w, p):
    return w / ((p["delta"].float()[..., None] * p["s"].float()) * p["sr"].float()[:, None, None]) + \
        p["zu"].float()[..., None]


def _grads(w, p, codes, G, element=False):
    """Gradients of the FlexRound-transformed quantizer; p in 64 bits, grouped."""
    f = _filter(_x32(w, p), p["alpha"], p["zb"], codes)
    d, zu, sr = p["delta"][..., None], p["zu"][..., None], p["sr"][:, None, None]
    u = w.double() / (d * p["s"] * sr)
    m = _value(p["alpha"], p["zb"], codes)
    if element:
        G = G * f
    return {"dalpha": p["delta"][..., None] * _dalpha(G, codes, p["alpha"].shape[-1]),
            "ddelta": (G * (m - zu - f * u)).sum(-1), "ds": -G * d * f * u / p["s"],
            "dsr": -(G * d * f * u).sum((-1, -2)) / p["sr"], "dzb": (G * d).sum(-1),
            "dzu": (G * d * (f - 1.0)).sum(-1)}


def _omni_scales(wg, p, q):
    lo, hi = wg.amin(-1), wg.amax(-1)
    delta = (p["gamma"] * hi - p["beta"] * lo) / torch.full_like(hi, 2 ** q - 1)   # a scalar divisor is inverted first
    return delta, -torch.round((p["beta"] * lo) / delta)


def _rows(case):
    step = max(1, CHUNK // case["n_in"])
    return [slice(r, min(r + step, case["out"])) for r in range(0, case["out"], step)]


def _cat(parts):
    if isinstance(parts[0], dict):
        return {k: _cat([p[k] for p in parts]) for k in parts[0]}
    return None if parts[0] is None else torch.cat(parts)


def _take(p, r, g):
    """The rows r of the parameters in 64 bits, s grouped."""
    return {k: (_groups(v[r], g) if k == "s" else v[r]).double() for k, v in p.items()}


def exact(case, seed):
    st = prepare(case, seed)
    kind, q, g, n_in = case["kind"], case["q"], case["g"], case["n_in"]
    if kind == "product":
        parts = []
        for r in _rows(case):
            bits = (st["planes"][:, r, :, None] >> torch.arange(32, device="cuda", dtype=torch.int32)) & 1
            c = _groups(bits.reshape(-1, n_in), g).reshape(q, -1, n_in // g, g).double().mul_(2).sub_(1)
            w = torch.einsum("qrkg,rkq->rkg", c, st["alpha"][r].double()) + st["zb"][r].double()[..., None]
            parts.append(st["x"].double() @ w.reshape(-1, n_in).T)
        return torch.cat(parts, 1)
    if kind == "export":
        p = st["params"]
        return {"alpha": p["delta"].double()[..., None] * p["alpha"].double(), "planes": None,
                "zb": p["delta"].double() * (p["zb"].double() - p["zu"].double())}
    flat = lambda t: t.reshape(t.shape[0], n_in)  # noqa: E731
    parts = []
    dsa = torch.zeros(n_in, dtype=torch.float64, device="cuda")
    for r in _rows(case):
        w = _groups(st["W"][r], g).float()
        if kind == "init":
            parts.append(_init(w, q))
            continue
        codes = _groups(st["codes"][r], g).long()
        G = _groups(st["grad"][r], g).double()
        res = {"codes": None}
        if kind == "step":
            for i, (_, p, _, _) in enumerate(st["steps"]):
                p = _take(p, r, g)
                mode = "full" if case["map"] == "full" else ("remap", "keep")[i]
                codes = _map(_x32(w, p), p["alpha"], p["zb"], codes, mode)
                res["what%d" % i] = flat(p["delta"][..., None] * (_value(p["alpha"], p["zb"], codes) - p["zu"][..., None]))
                gr = _grads(w, p, codes, G, case["filter"] == "element")
                res["grads%d" % i] = dict(gr, ds=flat(gr["ds"]))
        elif kind == "fused":
            p = _take(st["params"], r, g)
            for i in range(2):
                gr = _grads(w, p, codes, G)
                p = {k: v - (LR_B if k in ("alpha", "zb") else LR_F) * gr["d" + k] for k, v in p.items()}
                codes = _map(_x32(w, p), p["alpha"], p["zb"], codes, ("keep", "remap")[i])
                res["what%d" % i] = flat(p["delta"][..., None] * (_value(p["alpha"], p["zb"], codes) - p["zu"][..., None]))
            res["params"] = dict(p, s=flat(p["s"]))
        else:
            p32 = {k: (v if k == "sa" else v[r]) for k, v in st["params"].items()}
            p = {k: v.double() for k, v in p32.items()}
            col = _groups(p32["sa"][None], g) if kind == "awq" else 1.0
            d32, z32 = (p32["delta"], p32["za"]) if kind == "awq" else _omni_scales(w, p32, q)
            d, z = (p["delta"], p["za"]) if kind == "awq" else _omni_scales(w.double(), p, q)
            z = z32.double()                           # OmniQuant's is a whole number: a decision
            x32 = (w * col) / d32[..., None] + z32[..., None]
            scol = col.double() if kind == "awq" else 1.0
            for i in range(2):
                codes = _map(x32, p["alpha"], p["zb"], codes, ("remap", "keep")[i])
                res["what%d" % i] = flat(d[..., None] * (_value(p["alpha"], p["zb"], codes) - z[..., None]) / scol)
            f = _filter(x32, p["alpha"], p["zb"], codes)
            m = _value(p["alpha"], p["zb"], codes) - z[..., None]
            u = w.double() * scol / d[..., None]
            Gs = G / scol
            A, B = (Gs * (m - f * u)).sum(-1), -d * (Gs * (1.0 - f)).sum(-1)
            gr = {"dalpha": d[..., None] * _dalpha(Gs, codes, q), "dzb": d * Gs.sum(-1)}
            if kind == "awq":
                dsa += (Gs * (f * w.double() - d[..., None] * m / scol)).sum(0).reshape(-1)
                gr.update(ddelta=A, dza=B)
            else:
                lo, hi, top = w.amin(-1).double(), w.amax(-1).double(), float(2 ** q - 1)
                db, dg = -lo / top, hi / top
                zb_, zg_ = -(lo / d - p["beta"] * lo * db / d ** 2), p["beta"] * lo * dg / d ** 2
                gr.update(dbeta=A * db + B * zb_, dgamma=A * dg + B * zg_)
            res["grads"] = gr
        parts.append(res)
    res = _cat(parts)
    if kind == "awq":
        res["grads"]["dsa"] = dsa
    return res


def _init(w, q):
    """Unified initialization of the groups of some rows, fixed-minimum clipping, G > 1 (z_B stays)."""
    shape, g = w.shape[:2], w.shape[2]
    n = w.shape[0] * w.shape[1]
    top = torch.full((n,), float(2 ** q - 1), device="cuda")
    w = w.reshape(n, g)
    lo = w.amin(-1)
    span = (w.amax(-1) - lo).clamp_min(1e-12)
    zb = top * 0.5
    signs = _signs(q)
    best = {"e": torch.full((n,), math.inf, dtype=torch.float64, device="cuda")}
    for i in range(1, INIT_G + 1):
        gamma = torch.full_like(span, float(i)) / torch.full_like(span, float(INIT_G))
        d = (gamma * span) / top
        zu = -lo / d
        x = w / d[:, None] + zu[:, None]
        r, codes, alpha = x - zb[:, None], torch.zeros(n, g, dtype=torch.int64, device="cuda"), []
        for j in range(q):
            up = r >= 0
            codes += up.long() << j
            a = (r.abs().double().sum(-1) / g).float()
            alpha.append(a)
            r = r - torch.where(up, a[:, None], -a[:, None])
        alpha = torch.stack(alpha, -1)
        y = x.double() - zb.double()[:, None]
        for _ in range(INIT_T):
            C = torch.gather(signs[None].expand(n, -1, -1), 2, codes[:, None].expand(-1, q, -1))
            M, b = C @ C.transpose(1, 2), (C * y[:, None]).sum(-1)
            ok = torch.linalg.det(M).abs() > 0.5       # whole numbers: singular means zero
            M = torch.where(ok[:, None, None], M, torch.eye(q, dtype=torch.float64, device="cuda"))
            new = torch.linalg.solve(M, b).float()
            alpha = torch.where(ok[:, None], new, alpha)
            codes = _nearest(x, _levels32(alpha, zb))
        lv = torch.gather(_levels32(alpha, zb), -1, _nearest(x, _levels32(alpha, zb)))
        what = d[:, None] * (lv - zu[:, None])
        e = (w.double() - what.double()).square().sum(-1)
        take = e < best["e"]
        for k, v in {"e": e, "delta": d, "zu": zu, "alpha": alpha}.items():
            t = take.reshape(n, *([1] * (v.dim() - 1)))
            best[k] = torch.where(t, v, best[k]) if k in best else v.clone()
    rows = {k: best[k].double().reshape(*shape, *best[k].shape[1:]) for k in ("alpha", "delta", "zu")}
    rows["s"] = torch.ones(shape[0], shape[1] * g, dtype=torch.float64, device="cuda")
    rows["sr"] = torch.ones(shape[0], dtype=torch.float64, device="cuda")
    rows["zb"] = zb.double().reshape(shape)
    return {"codes": None, "params": rows}
