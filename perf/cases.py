"""Performance cases of the DendSN and LIF layers.

A case is one pass through the library's public entry points (paper_2412_06355_gb300.binding):
a training step of a layer (forward and BPTT backward, with every gradient it returns) or a
forward alone. Layer shapes and value distributions are those of the package's workloads
(workloads.py), of the paper's networks (T = 6 and 10, P = 4 compartments on 2 branches, the
(C_o, P, H, W) layout) and generic ones in between.

Fields of a case:
  op       "dendsn" or "lif" (the point-neuron layer)
  mode     "train": forward and backward; "infer": the forward alone, with V^s
  api      "abi": the C-ABI calls on buffers the program keeps; "autograd": DendSNFunction
           with a layer-wide alpha
  T, B, C, inner, rep   time steps, samples, channels, neurons per channel run, and how often
           the C * inner pattern repeats in a sample (tokens); N = C * inner * rep
  K, G     compartments per neuron, compartments per branch
  dtype, psi, reset, beta, detach, stateless, residual, layout, plif   as in dendsn_config;
           plif: dL/dbeta is wanted too
  mask     "none", "channel" or "neuron" (Bernoulli(0.5) branch gating)
  x_mean, x_std, density   inputs: N(x_mean, x_std) times Bernoulli(density)
"""
import math

import torch

from paper_2412_06355_gb300 import binding

BASE = dict(op="dendsn", mode="train", api="abi", T=4, B=64, C=128, inner=1024, rep=1, K=4, G=1,
            dtype="f32", psi="mh", reset="hard", beta=0.5, detach=False, stateless=False,
            residual=False, layout="kinner", plif=False, mask="none", x_mean=0.3, x_std=1.0,
            density=1.0)


def case(name, **kw):
    return dict(BASE, name=name, **kw)


def listed():
    return [
        # the smallest layer, as a training program calls it: latency and launches count
        case("tiny", api="autograd", B=2, C=64, inner=1),
        # a VGG conv layer at CIFAR / Tiny ImageNet scale, float32
        case("conv"),
        # the same layer as the conv kernel leaves it, P = 4 compartments on 2 branches
        case("conv_paper_p4b2", G=2, layout="paper"),
        # mixed-precision training of the paper's Tiny ImageNet network: T = 6, batch 128,
        # the ResStateless dendrite, straight from a bfloat16 conv output
        case("vgg_bf16", T=6, B=128, G=2, dtype="bf16", stateless=True, residual=True,
             layout="paper"),
        # a deeper conv layer with bfloat16 currents, 8 compartments, soft reset
        case("deepconv_bf16", T=8, B=128, C=256, inner=256, K=8, dtype="bf16", reset="soft"),
        # a long event stream (DVS-like): sparse float32 input; the largest case
        case("event", T=64, B=32, x_mean=0.8, density=0.2),
        # a transformer layer (196 tokens x 384 features) with per-neuron branch gating
        case("token_dbg", C=384, inner=1, rep=196, K=8, mask="neuron"),
        # the single-neuron fit over a 2048-step horizon
        case("l5pc", T=2048, B=16, C=1, inner=1, G=2, beta=0.95, x_mean=0.1, x_std=0.5,
             density=0.3),
        # the same horizon on a layer
        case("long_t", T=2048, B=16, C=4, inner=1024, G=2, beta=0.95, x_mean=0.1, x_std=0.5,
             density=0.3),
        # a late layer of a CIFAR10-DVS-like network: T = 10, 7 x 7 positions (no multiple of
        # a warp), the Stateless dendrite, a learnable somatic decay
        case("dvs_plif", T=10, B=32, C=512, inner=49, G=2, stateless=True, layout="paper",
             plif=True),
        # inference at a small batch: 14 x 14 positions, bfloat16, the potentials read out
        case("infer_bf16", mode="infer", T=6, B=16, C=256, inner=196, G=2, dtype="bf16",
             layout="paper"),
        # the point-neuron layer the DendSN layers are compared with
        case("lif", op="lif", x_mean=0.5),
    ]


# ---------------------------------------------------------------- sizes
def neurons(c):
    return c["C"] * c["inner"] * c["rep"]


def elem(c):
    return 2 if c["dtype"] == "bf16" else 4


def work(c):
    ns, s = c["T"] * c["B"] * neurons(c), elem(c)
    train = c["mode"] == "train"
    if c["op"] == "lif":                       # x, S; dL/dS, dL/dX
        return {"bytes": ns * s * (4 if train else 2) + (0 if train else 4 * ns),
                "flops": ns * (2 + (9 if train else 0))}
    K, Kb = c["K"], c["K"] // c["G"]
    par = 4 * c["C"] * 2 * (K + Kb) * (2 if train else 1)
    if c["mask"] != "none":
        par += (c["C"] if c["mask"] == "channel" else neurons(c)) * Kb
    # each input once (x, dL/dS), each output once (S or V^s too, dL/dX)
    b = ns * (K * s + s) + (ns * (K * s + s) if train else 4 * ns) + par
    # fused multiply-adds counted as two; transcendentals as one
    f = 6 * K + 6 * Kb + 4
    if train:
        f += 12 * K + 16 * Kb + 14
    return {"bytes": b, "flops": ns * f}


MAX_BYTES = 8.0e9                              # drawn cases stay below the largest listed one


def draw(rng):
    kind = rng.choice(["conv", "conv", "conv", "token", "fc", "events", "long", "lif"])
    c = dict(BASE)
    log = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    c["dtype"] = rng.choice(["f32", "f32", "bf16"])
    c["mode"] = "train" if rng.random() < 0.8 else "infer"
    c["reset"] = rng.choice(["hard", "hard", "soft"])
    c["psi"] = rng.choice(["mh", "mh", "mh", "identity"])
    c["K"], c["G"] = rng.choice([(4, 1), (4, 2), (4, 2), (8, 1), (8, 2), (2, 1), (16, 2), (1, 1)])
    if kind != "lif" and c["mode"] == "train":
        c["plif"] = rng.random() < 0.15
    c["detach"] = rng.random() < 0.1
    variant = rng.random()
    c["stateless"] = variant < 0.3
    c["residual"] = variant < 0.15 or variant > 0.85
    c["mask"] = rng.choice(["none", "none", "none", "channel"])
    c["T"] = rng.choice([1, 2, 4, 4, 4, 5, 6, 6, 8, 8, 10, 16])
    c["B"] = log(1, 128)
    if kind in ("conv", "lif"):
        side = rng.choice([4, 7, 8, 14, 16, 28, 32, 56, 64])
        c["inner"] = side * side
        c["C"] = rng.choice([10, 64, 96, 128, 192, 256, 512])
        c["layout"] = rng.choice(["paper", "paper", "kinner"])
    elif kind == "token":
        c["C"], c["inner"], c["rep"] = rng.choice([192, 384, 768]), 1, rng.choice([50, 196, 197])
        c["mask"] = rng.choice(["none", "neuron", "neuron"])
    elif kind == "fc":
        c["C"], c["inner"] = log(10, 4096), 1
        c["api"] = rng.choice(["abi", "autograd"]) if c["mode"] == "train" else "abi"
    elif kind == "events":
        c["T"] = log(10, 128)
        side = rng.choice([4, 8, 16, 32])
        c["inner"], c["C"] = side * side, rng.choice([64, 128, 256])
        c["B"] = log(1, 32)
        c["layout"] = rng.choice(["paper", "kinner"])
        c["x_mean"], c["density"] = 0.8, 0.2
    else:                                      # "long": few neurons, a long horizon
        c["T"] = log(256, 2048)
        c["C"], c["inner"] = rng.choice([(1, 1), (1, 8), (4, 64), (10, 100)])
        c["B"] = log(1, 32)
        c["beta"], c["x_mean"], c["x_std"], c["density"] = 0.95, 0.1, 0.5, 0.3
        c["mask"] = "none"
    if kind == "lif":
        c["op"], c["layout"], c["x_mean"], c["K"], c["G"] = "lif", "kinner", 0.5, 1, 1
        c["plif"] = c["stateless"] = c["residual"] = False
        c["psi"], c["mask"] = "mh", "none"
    if c["api"] == "autograd":
        c["dtype"] = "f32"
    while work(c)["bytes"] > MAX_BYTES:
        if c["B"] > 1:
            c["B"] = (c["B"] + 1) // 2
        else:
            c["C"] = (c["C"] + 1) // 2
    return c


# ---------------------------------------------------------------- inputs
def inputs(c, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    f32 = dict(generator=g, dtype=torch.float32, device="cuda")
    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    T, B, N, K, C = c["T"], c["B"], neurons(c), c["K"], c["C"]
    Kb = K // c["G"]
    if c["op"] == "lif":
        shape = (T, B, N)
    elif c["layout"] == "paper":
        shape = (T, B, N // c["inner"], K, c["inner"])
    else:
        shape = (T, B, N, K)
    x = torch.randn(shape, **f32).mul_(c["x_std"]).add_(c["x_mean"])
    if c["density"] < 1.0:
        x.mul_(torch.rand(shape, **f32) < c["density"])
    d = dict(x=x.to(dt), gs=torch.randn((T, B, N), **f32).to(dt))
    if c["op"] == "lif":
        return d
    if c["api"] == "autograd":
        d["alpha"] = torch.rand((), **f32).mul_(0.45).add_(0.5)
    else:
        d["alpha"] = torch.rand((C, K), **f32).mul_(0.45).add_(0.5)
    d["xi"] = torch.randn((C, K), **f32).mul_(0.1)
    d["zeta"] = torch.rand((C, Kb), **f32).mul_(0.4).add_(0.8)
    d["kappa"] = torch.randn((C, Kb), **f32).mul_(0.1).add_(1.0 / K)
    d["mask"] = None
    if c["mask"] != "none":
        rows = N if c["mask"] == "neuron" else C
        d["mask"] = (torch.rand((rows, Kb), **f32) < 0.5).to(torch.uint8)
    return d


def prepare(c, seed):
    d = inputs(c, seed)
    T, B, N, K, C = c["T"], c["B"], neurons(c), c["K"], c["C"]
    st = dict(case=c, **d)
    x = d["x"]
    st["s"] = torch.empty((T, B, N), dtype=x.dtype, device="cuda")
    if c["mode"] == "infer":
        st["v"] = torch.empty((T, B, N), dtype=torch.float32, device="cuda")
    if c["op"] == "lif":
        st["cfg"] = binding.make_lif_config(T, B, N, c["dtype"], c["reset"], beta=c["beta"],
                                            detach_reset=c["detach"])
        st["saved"] = binding.lif_workspace(st["cfg"])
        st["gx"] = torch.empty_like(x)
        return st
    st["cfg"] = binding.make_config(T, B, N, K, c["G"], C, c["inner"], c["dtype"], c["psi"],
                                    c["reset"], beta=c["beta"], detach_reset=c["detach"],
                                    mask_per_neuron=c["mask"] == "neuron",
                                    stateless=c["stateless"], residual=c["residual"],
                                    layout=c["layout"])
    if c["api"] == "autograd":
        for k in ("x", "alpha", "xi", "zeta", "kappa"):
            st[k].requires_grad_(True)
        st["beta"] = (torch.tensor(c["beta"], device="cuda", requires_grad=True)
                      if c["plif"] else None)
    elif c["mode"] == "train":
        st["saved"], st["scratch"] = binding.workspace(st["cfg"])
        st["gx"] = torch.empty_like(x)
        for k in ("alpha", "xi", "zeta", "kappa"):
            st["g" + k] = torch.empty_like(d[k])
        if c["plif"]:
            st["gbeta"] = torch.empty((C,), dtype=torch.float32, device="cuda")
    return st


def run(st):
    c, cfg = st["case"], st["cfg"]
    train = c["mode"] == "train"
    if c["op"] == "lif":
        if not train:
            binding.dendsn_lif_forward(cfg, st["x"], st["s"], st["v"])
            return {"s": st["s"], "v": st["v"]}
        binding.dendsn_lif_forward(cfg, st["x"], st["s"], None, st["saved"])
        binding.dendsn_lif_backward(cfg, st["x"], st["gs"], None, st["saved"], st["gx"])
        return {"s": st["s"], "gx": st["gx"]}
    if c["api"] == "autograd":
        leaves = [st[k] for k in ("x", "alpha", "xi", "zeta", "kappa")]
        s = binding.DendSNFunction.apply(*leaves, st["mask"], cfg, st["beta"])
        if c["plif"]:
            leaves.append(st["beta"])
        g = torch.autograd.grad(s, leaves, st["gs"])
        return dict(zip(("s", "gx", "galpha", "gxi", "gzeta", "gkappa", "gbeta"), (s, *g)))
    p = (st["x"], st["alpha"], st["xi"], st["zeta"], st["kappa"], st["mask"])
    if not train:
        binding.dendsn_forward(cfg, *p, st["s"], st["v"])
        return {"s": st["s"], "v": st["v"]}
    binding.dendsn_forward(cfg, *p, st["s"], None, st["saved"])
    grads = [st["g" + k] for k in ("alpha", "xi", "zeta", "kappa")]
    out = {"s": st["s"], "gx": st["gx"]}
    out.update({"g" + k: st["g" + k] for k in ("alpha", "xi", "zeta", "kappa")})
    if c["plif"]:
        binding.dendsn_backward_plif(cfg, *p, st["gs"], None, st["saved"], st["gx"], *grads,
                                     st["gbeta"], st["scratch"])
        out["gbeta"] = st["gbeta"]
    else:
        binding.dendsn_backward(cfg, *p, st["gs"], None, st["saved"], st["gx"], *grads,
                                st["scratch"])
    return out


# ---------------------------------------------------------------- float64 values
def exact(c, seed):
    """The layer's equations and their chain rule in float64, step by step."""
    d = inputs(c, seed)
    T, B, N, K, C, G = c["T"], c["B"], neurons(c), c["K"], c["C"], c["G"]
    lif, train, soft = c["op"] == "lif", c["mode"] == "train", c["reset"] == "soft"
    Kb, theta = K // G, 1.0
    beta = float(torch.tensor(c["beta"], dtype=torch.float32))
    f64 = dict(dtype=torch.float64, device="cuda")
    row = (B, c["rep"], C, c["inner"])         # a step's neurons; channel axis 2
    if lif:
        xs = d["x"].view(T, *row)
        step_x = lambda t: xs[t].double()
    else:
        if c["layout"] == "paper":
            xs = d["x"].view(T, B, c["rep"], C, K, c["inner"]).transpose(-1, -2)
        else:
            xs = d["x"].view(T, *row, K)
        step_x = lambda t: xs[t].double()
        par = lambda p: p.double().view(C, 1, -1)
        alpha = d["alpha"].double().expand(C, K).reshape(C, 1, K)
        xi, zeta, kappa = par(d["xi"]), par(d["zeta"]), par(d["kappa"])
        zeta_k = zeta.repeat_interleave(G, -1)
        m = 1.0
        if d["mask"] is not None:
            m = d["mask"].double()
            m = m.view(C, 1, Kb) if c["mask"] == "channel" else m.view(c["rep"], C, c["inner"], Kb)

    def branches(vd):
        u = (vd - xi) / zeta_k
        q = (u * u).view(*row, Kb, G).sum(-1)
        if c["psi"] == "mh":
            e = torch.exp(-0.5 * q)
            return u, (1.0 - q) * e, (q - 3.0) * e          # psi, psi'(r) / r
        r = q.sqrt()
        return u, r, torch.where(r > 0, 1.0 / r, torch.zeros_like(r))

    s_all = torch.empty((T, *row), **f64)
    v_all = torch.empty((T, *row), **f64)
    hist = []
    v, s = torch.zeros(row, **f64), torch.zeros(row, **f64)
    vd = None if lif else torch.zeros((*row, K), **f64)
    for t in range(T):
        x = step_x(t)
        if lif:
            z = x
        else:
            vd = x if c["stateless"] else alpha * vd + x
            if train:
                hist.append(vd)
            z = (kappa * m * branches(vd)[1]).sum(-1)
            if c["residual"]:
                z = z + x.mean(-1)
        v = beta * (v - theta * s if soft else v * (1.0 - s)) + z
        s = (v >= theta).double()
        s_all[t], v_all[t] = s, v
    out = {"s": s_all.view(T, B, N)}
    if not train:
        out["v"] = v_all.view(T, B, N)
        return out

    gs = d["gs"].view(T, *row)
    dvn = torch.zeros(row, **f64)
    gbeta = torch.zeros(C, **f64)
    gx = torch.empty(d["x"].shape, **f64)
    if lif:
        gx_t = gx.view(T, *row)
    else:
        if c["layout"] == "paper":
            gx_t = gx.view(T, B, c["rep"], C, K, c["inner"]).transpose(-1, -2)
        else:
            gx_t = gx.view(T, *row, K)
        A = torch.zeros((*row, K), **f64)
        galpha, gxi = torch.zeros((C, K), **f64), torch.zeros((C, K), **f64)
        gzeta, gkappa = torch.zeros((C, Kb), **f64), torch.zeros((C, Kb), **f64)
    per_channel = lambda q: q.sum(dim=(0, 1, 3))
    for t in range(T - 1, -1, -1):
        v, s = v_all[t], s_all[t]
        if c["plif"]:
            gbeta += per_channel((dvn * (v - theta * s if soft else v * (1.0 - s))).unsqueeze(-1))[:, 0]
        ds = gs[t].double()
        if not c["detach"]:
            ds = ds - beta * (theta if soft else v) * dvn
        sg = 1.0 / (1.0 + math.pi ** 2 * (v - theta) ** 2)
        dvn = sg * ds + beta * (1.0 if soft else (1.0 - s)) * dvn
        if lif:
            gx_t[t] = dvn
            continue
        dz = dvn.unsqueeze(-1)
        u, y, w = branches(hist[t])
        gkappa += per_channel(m * y * dz)
        du = (kappa * m * dz * w).repeat_interleave(G, -1) * u
        gzeta -= per_channel(((du * u).view(*row, Kb, G).sum(-1)) / zeta)
        direct = du / zeta_k
        gxi -= per_channel(direct)
        if c["stateless"]:
            A = direct
        else:
            A = direct + alpha * A
            if t > 0:
                galpha += per_channel(A * hist[t - 1])
        hist[t] = None                         # free as the sweep goes
        gx_t[t] = A + dz / K if c["residual"] else A
    out["gx"] = gx
    if not lif:
        out.update(galpha=galpha.sum() if c["api"] == "autograd" else galpha, gxi=gxi,
                   gzeta=gzeta, gkappa=gkappa)
        if c["plif"]:
            out["gbeta"] = gbeta.sum() if c["api"] == "autograd" else gbeta
    return out
