"""The work that a user of this library has it do, as measurable cases.

A verification run bounds one robustness property (or a batch of them) of a
ReLU convnet: interval or CROWN/WK intermediate bounds of the root, LD bounds
of a batch of branch-and-bound subdomains (FP32 or BF16 iterations, FP64
final bound), the branching decision for the next batch, bounds recomputed
per subdomain, the proximal solver as the alternative ascent; certified
training adds the Danskin gradients through torch.autograd.  The nets are the
repository's own (tiny MLP, Base, Wide, Deep), the batch sizes and iteration
counts those of its benchmark, its Deep sweep (64-8192 subdomains, 32
properties, 50-500 iterations) and its branch and bound.

Inputs are drawn on their own here (Kaiming weights, images U[0,1], boxes of
radius 1/255 to 8/255, splits of root-ambiguous ReLUs); intermediate bounds
handed to the solvers are interval bounds rounded outward to FP32.  Iterated
solvers name their engine and launch shape (as the branch-and-bound driver
does), so that a run does not depend on the autotuner's timing.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2104_06718_gb300 import autograd as ld_autograd
from paper_2104_06718_gb300 import binding as ld
from paper_2104_06718_gb300.synth import LayerSpec

# (cout, k, stride, pad) per conv, then FC widths (10 logits); input 3x32x32
CONVNETS = {
    "base": ([(8, 4, 2, 1), (16, 4, 2, 1)], [100, 10]),
    "wide": ([(16, 4, 2, 1), (32, 4, 2, 1)], [100, 10]),
    "deep": ([(8, 4, 2, 1), (8, 3, 1, 1), (8, 3, 1, 1), (8, 4, 2, 1)], [100, 10]),
}
TINY = [10, 20, 20, 1]
ETA = (10.0, 500.0, 0.3, 2)      # proximal solver: eta first / last, momentum, sweeps (the library's defaults)
TIE = 2.0 ** -16                 # tie margin of the library's vertex choice


def listed():
    return [
        # the smallest solve: one property of a small MLP, latency only
        dict(name="tiny_fp32", kind="bound", net="tiny", B=1, P=1, T=200, precision="fp32", tile=1),
        # the headline: a branch-and-bound batch of 256 subdomains, FP32 and BF16 iterations
        dict(name="base256_fp32", kind="bound", net="base", B=256, P=1, T=100, precision="fp32", tile=2),
        dict(name="base256_bf16", kind="bound", net="base", B=256, P=1, T=100, precision="bf16", tile=2),
        # the large batch: 2048 subdomains of the Wide net, BF16 layer-wise tensor-core engine
        dict(name="wide2048_bf16", kind="bound", net="wide", B=2048, P=1, T=100, precision="bf16", tile=0),
        # the Deep sweep: 32 properties in one batch, FP32
        dict(name="deep1024_fp32", kind="bound", net="deep", B=1024, P=32, T=50, precision="fp32", tile=1),
        # one step of certified training: bounds and their gradients (weights, biases, boxes, bounds)
        dict(name="deep128_grad", kind="grad", net="deep", B=128, P=1, T=20, precision="fp32", tile=1),
        # root interval bounds of a batch of properties: the cheapest call of a run
        dict(name="deep32_interval", kind="interval", net="deep", P=32),
        # root bounds of one property, layer-wise best of CROWN and WK: what a run starts with
        dict(name="deep1_root", kind="propagated", net="deep", B=0, P=1),
        # the same recomputed per subdomain after its splits
        dict(name="base64_split", kind="propagated", net="base", B=64, P=1),
        # the proximal solver on a branch-and-bound batch
        dict(name="base256_proximal", kind="proximal", net="base", B=256, P=1, T=100),
        # filtered smart branching decisions of a batch
        dict(name="base256_fsb", kind="fsb", net="base", B=256, P=1),
        # dual value, supergradient and upper bounds at given duals: the evaluation calls of a custom ascent or search
        dict(name="wide512_eval", kind="eval", net="wide", B=512, P=1),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    most = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(["bound", "bound", "bound", "grad", "interval", "propagated", "propagated", "proximal", "fsb", "eval"])
        net = rng.choice(["base", "wide", "deep"])
        c = dict(kind=kind, net=net)
        if kind == "bound":
            c["precision"] = rng.choice(["fp32", "bf16"])
            if c["precision"] == "fp32" and rng.random() < 0.2:
                c["net"] = "tiny"
            c |= dict(B=log(1, 2048), T=log(10, 200))
            c["P"] = min(c["B"], rng.choice([1, 1, log(2, 32)]))
            # tile 0: the layer-wise engine (large BF16 batches)
            large = c["precision"] == "bf16" and c["B"] >= 1024
            c["tile"] = 0 if large else 1 if c["B"] <= 152 or c["net"] != "base" else 2
        elif kind == "grad":
            c |= dict(B=log(8, 256), P=1, T=log(5, 40), precision="fp32", tile=1)
        elif kind == "interval":
            c |= dict(P=log(1, 256))
        elif kind == "propagated":
            c |= dict(B=0, P=log(1, 8)) if rng.random() < 0.4 else dict(B=log(2, 64), P=1)
        elif kind == "proximal":
            c |= dict(B=log(4, 512), P=1, T=log(5, 100))
        elif kind == "fsb":
            c |= dict(B=log(2, 256), P=1)
        else:
            c |= dict(B=log(1, 1024), P=1)
        if _cost(c) <= most:
            return c


# ------------------------------------------------------------------ inputs

class _Inputs:
    """Net, boxes, interval bounds and splits of a case (float32, on the GPU), from its seed."""

    def __init__(self, case, seed):
        rng = np.random.default_rng([int(seed), 1])
        gen = torch.Generator("cuda").manual_seed(int(seed))
        self.layers = _layers(case["net"], rng)
        self.margin = None
        P, n0 = case["P"], int(np.prod(self.layers[0].in_shape))
        if case["net"] == "tiny":
            x = rng.uniform(-1.0, 1.0, (P, n0))
            eps = np.full((P, 1), 0.1)
        else:
            x = rng.uniform(0.0, 1.0, (P, n0))
            eps = rng.uniform(1 / 255, 8 / 255, (P, 1))
            gt, other = rng.choice(10, 2, replace=False)
            self.margin = np.zeros(10, np.float32)
            self.margin[gt], self.margin[other] = 1.0, -1.0
        self.l0 = torch.as_tensor((x - eps).astype(np.float32), device="cuda")
        self.u0 = torch.as_tensor((x + eps).astype(np.float32), device="cuda")
        self.ref = _Net64(self.layers, self.margin)
        lb, ub = self.ref.interval(self.l0.double(), self.u0.double())
        inf = torch.tensor(math.inf, device="cuda")
        self.lbk = torch.nextafter(lb.float(), -inf)
        self.ubk = torch.nextafter(ub.float(), inf)
        B = case.get("B", 0)
        self.prop = self.masks = None
        if B:
            if P > 1:
                self.prop = torch.arange(B, device="cuda", dtype=torch.int32) * P // B
            # split depth 0-8 (Wide: 0-20) on ReLUs ambiguous at the root of property 0; subdomain 0 is the root
            amb = torch.nonzero((self.lbk < 0).all(0) & (self.ubk > 0).all(0)).reshape(-1)
            most = min(20 if case["net"] == "wide" else 8, amb.numel())
            self.masks = torch.zeros((B, self.ref.N), dtype=torch.int8, device="cuda")
            if most:
                col = torch.rand((B, amb.numel()), device="cuda", generator=gen).topk(most, dim=1).indices
                depth = torch.randint(0, most + 1, (B, 1), device="cuda", generator=gen)
                depth[0] = 0
                sign = 2 * torch.randint(0, 2, (B, most), device="cuda", generator=gen) - 1
                keep = torch.arange(most, device="cuda")[None] < depth
                self.masks.scatter_(1, amb[col], (sign * keep).to(torch.int8))
        if case["kind"] == "eval":
            # duals of an ascent under way: the CROWN start moved by a few Adam steps' worth
            lo, up = self.clamped()
            rho = torch.cat(self.ref.crown(lo, up)[0], 1)
            rho = rho + 0.05 * torch.randn(rho.shape, device="cuda", generator=gen, dtype=torch.float64)
            self.rho = rho.float()

    def clamped(self):
        """Bounds per subdomain after its splits, float64 [B, N]."""
        row = torch.zeros(self.masks.shape[0], dtype=torch.long, device="cuda") if self.prop is None else self.prop.long()
        lo, up = self.lbk.double()[row], self.ubk.double()[row]
        lo = torch.where(self.masks > 0, lo.clamp(min=0), lo)
        return lo, torch.where(self.masks < 0, up.clamp(max=0), up)

    def boxes(self):
        row = torch.zeros(self.masks.shape[0], dtype=torch.long, device="cuda") if self.prop is None else self.prop.long()
        return self.l0.double()[row], self.u0.double()[row]


def _layers(net, rng):
    out = []
    if net == "tiny":
        for a, b in zip(TINY[:-1], TINY[1:]):
            W, bias = rng.normal(0, math.sqrt(1 / a), (b, a)), rng.normal(0, 0.1, b)
            out.append(LayerSpec("fc", W.astype(np.float32), bias.astype(np.float32), (a,)))
        return out
    convs, fcs = CONVNETS[net]
    shape = (3, 32, 32)
    for cout, k, s, p in convs:
        fan = shape[0] * k * k
        W = rng.normal(0, math.sqrt(2 / fan), (cout, shape[0], k, k))
        bias = rng.uniform(-1 / math.sqrt(fan), 1 / math.sqrt(fan), cout)
        out.append(LayerSpec("conv", W.astype(np.float32), bias.astype(np.float32), shape, s, p))
        shape = (cout, (shape[1] + 2 * p - k) // s + 1, (shape[2] + 2 * p - k) // s + 1)
    n = int(np.prod(shape))
    for m in fcs:
        W = rng.normal(0, math.sqrt(2 / n), (m, n))
        bias = rng.uniform(-1 / math.sqrt(n), 1 / math.sqrt(n), m)
        out.append(LayerSpec("fc", W.astype(np.float32), bias.astype(np.float32), (n,)))
        n = m
    return out


# ------------------------------------------------------------------ the calls

def _options(case):
    if case["tile"] == 0:
        return ld.Options(precision=case["precision"], engine="layerwise")
    return ld.Options(precision=case["precision"], engine="fused", tile=case["tile"], cta_threads=512)


def prepare(case, seed):
    i = _Inputs(case, seed)
    s = dict(case=case, net=ld.Net(i.layers, margin=i.margin), l0=i.l0, u0=i.u0, lbk=i.lbk, ubk=i.ubk, prop=i.prop,
             masks=i.masks)
    if case.get("B"):
        s["net"].reserve(case["B"])
    if case["kind"] in ("bound", "grad"):
        s["opts"] = _options(case)
    if case["kind"] == "grad":
        s["params"] = [torch.as_tensor(a, device="cuda").requires_grad_() for L in i.layers for a in (L.W, L.b)]
        for k in ("l0", "u0", "lbk", "ubk"):
            s[k].requires_grad_()
    if case["kind"] == "eval":
        s["rho"] = i.rho
    return s


def run(state):
    case, net = state["case"], state["net"]
    l0, u0, lbk, ubk, prop, masks = (state[k] for k in ("l0", "u0", "lbk", "ubk", "prop", "masks"))
    kind = case["kind"]
    if kind == "bound":
        out, rho = ld.ld_bound(net, l0, u0, lbk, ubk, prop, masks, n_iters=case["T"], opts=state["opts"], return_rho=True)
        return {"bound": out, "rho": rho}
    if kind == "grad":
        wrt = [l0, u0, lbk, ubk, *state["params"]]
        out = ld_autograd.bound(net, l0, u0, lbk, ubk, state["params"], prop, masks, n_iters=case["T"], opts=state["opts"])
        return {"bound": out.detach(), "grads": list(torch.autograd.grad(out.mean(), wrt))}
    if kind == "interval":
        lo, up, out = ld.ld_intermediate_bounds(net, l0, u0, want_output_lb=True)
        return {"lower": lo, "upper": up, "output": out}
    if kind == "propagated":
        lo, up = ld.ld_intermediate_bounds_propagated(net, l0, u0, rules="best", masks=masks, prop=prop)
        return {"lower": lo, "upper": up}
    if kind == "proximal":
        out, rho = ld.ld_bound_proximal(net, l0, u0, lbk, ubk, prop, masks, n_iters=case["T"], return_rho=True)
        return {"bound": out, "rho": rho}
    if kind == "fsb":
        dec, child = ld.ld_branch(net, l0, u0, lbk, ubk, prop, masks, rule="fsb", return_child_bounds=True)
        return {"decision": dec, "children": child}
    q, sg, vtx = ld.ld_dual_supergradient(net, l0, u0, lbk, ubk, state["rho"], prop, masks)
    ub, x0 = ld.ld_upper_bound(net, l0, u0, lbk, ubk, state["rho"], prop, masks, return_x0=True)
    return {"q": q, "supergradient": sg, "vertex": vtx, "upper": ub, "x0": x0}


# ------------------------------------------------------------------ work

def _shapes(net):
    """Per layer (cin, h, w, cout, ho, wo, taps, stride); the margin leaves one output."""
    if net == "tiny":
        return [(a, 1, 1, b, 1, 1, 1, 1) for a, b in zip(TINY[:-1], TINY[1:])]
    convs, fcs = CONVNETS[net]
    out, (c, h) = [], (3, 32)
    for cout, k, s, p in convs:
        ho = (h + 2 * p - k) // s + 1
        out.append((c, h, h, cout, ho, ho, k * k, s))
        c, h = cout, ho
    n = c * h * h
    for m in [*fcs[:-1], 1]:
        out.append((n, 1, 1, m, 1, 1, 1, 1))
        n = m
    return out


def _macs(S):
    return [cin * cout * ho * wo * taps for cin, _, _, cout, ho, wo, taps, _ in S]


def _substitution_macs(S, k):
    """Products of one objective row of layer k (1-based) substituted back to the input: the row of W_k is
    given; below it each layer costs what its window of nonzero coefficients reaches."""
    cin, h, w, _, ho, wo, taps, _ = S[k - 1]
    conv = taps > 1
    side = math.isqrt(taps) if conv else None           # window of nonzero coefficients on x_{k-1}; None: all of it
    total = 0
    for cin, h, w, cout, ho, wo, taps, stride in reversed(S[: k - 1]):
        reach = min(side, ho) if side is not None and taps > 1 else ho
        total += cout * reach * reach * cin * taps
        side = (reach - 1) * stride + math.isqrt(taps) if taps > 1 else None
    return total


def work(case):
    S = _shapes(case["net"])
    n0 = S[0][0] * S[0][1] * S[0][2]
    N = sum(s[3] * s[4] * s[5] for s in S[:-1])
    macs = _macs(S)
    W = sum(cin * cout * taps + cout for cin, _, _, cout, _, _, taps, _ in S)
    P, B, T = case["P"], case.get("B", 0), case.get("T", 0)
    kind = case["kind"]
    problem = 4 * W + 8 * P * (n0 + N) + B * N           # weights, boxes and bounds, split masks
    one = 2 * sum(macs[:-1])                             # one pass over the hidden layers
    if kind in ("bound", "proximal"):
        sweeps = T * (ETA[3] if kind == "proximal" else 1)
        return {"bytes": problem + B * (4 * N + 8), "flops": B * (2 * sweeps * one + one)}
    if kind == "grad":
        return {"bytes": problem + 4 * W + 8 * P * (n0 + N) + 8 * B, "flops": B * (2 * T * one + 3 * one)}
    if kind == "interval":
        return {"bytes": 4 * W + 8 * P * (n0 + N) + 8 * P, "flops": 2 * P * 2 * sum(macs)}
    if kind == "propagated":
        rows = max(B, P)
        sub = sum(4 * S[k - 1][3] * S[k - 1][4] * S[k - 1][5] * _substitution_macs(S, k) for k in range(2, len(S)))
        return {"bytes": 4 * W + 8 * P * n0 + B * N + 8 * rows * N, "flops": rows * 2.0 * sub}
    if kind == "fsb":
        children = B * 4 * (len(S) - 1)
        return {"bytes": problem + 4 * B + 8 * children, "flops": children * 2 * 2 * sum(macs[:-1]) + B * one}
    return {"bytes": problem + B * (4 * N + 4 * N + N + 4 * n0 + 16), "flops": B * 4 * one}


def _cost(case):
    w = work(case)
    return max(w["bytes"], w["flops"] / 50)


# ------------------------------------------------------------------ the same in 64 bits

class _Net64:
    """The net in canonical form (margin folded) in float64 torch, and the bounding arithmetic on it."""

    def __init__(self, specs, margin):
        t = lambda a: torch.as_tensor(np.asarray(a, np.float64), device="cuda")
        self.spec = specs
        self.W, self.b = [t(s.W) for s in specs], [t(s.b) for s in specs]
        if margin is not None:
            self.W[-1], self.b[-1] = (t(margin) @ self.W[-1])[None], (t(margin) @ self.b[-1])[None]
        self.n = len(specs)
        self.out = [s.out_shape for s in specs[:-1]] + [(1,)]
        self.width = [int(np.prod(o)) for o in self.out]
        self.N = sum(self.width[:-1])
        self.bias = [b if len(o) == 1 else b.repeat_interleave(o[1] * o[2]) for b, o in zip(self.b, self.out)]

    def cut(self, flat):
        return list(torch.split(flat, self.width[:-1], dim=1))

    def lin(self, k, x, W=None):
        s, W = self.spec[k], self.W[k] if W is None else W
        if s.kind == "fc":
            return x @ W.T
        return F.conv2d(x.reshape(-1, *s.in_shape), W, stride=s.stride, padding=s.pad).flatten(1)

    def tr(self, k, r):
        s = self.spec[k]
        if s.kind == "fc":
            return r @ self.W[k]
        left = s.in_shape[1] - ((self.out[k][1] - 1) * s.stride - 2 * s.pad + s.W.shape[2])
        return F.conv_transpose2d(r.reshape(-1, *self.out[k]), self.W[k], stride=s.stride, padding=s.pad,
                                  output_padding=left).flatten(1)

    def interval(self, lo, up, output=False):
        los, ups = [], []
        for k in range(self.n if output else self.n - 1):
            c, r = self.lin(k, (lo + up) / 2) + self.bias[k], self.lin(k, (up - lo) / 2, self.W[k].abs())
            los.append(c - r)
            ups.append(c + r)
            lo, up = (c - r).clamp(min=0), (c + r).clamp(min=0)
        if output:
            return torch.cat(los[:-1], 1), torch.cat(ups[:-1], 1), los[-1][:, 0]
        return torch.cat(los, 1), torch.cat(ups, 1)

    @staticmethod
    def relaxation(l, u, crown):
        """Lower slope, upper slope and upper intercept of a ReLU on [l, u]."""
        amb, on = (l < 0) & (u > 0), ((l >= 0) & (u > 0)).double()
        den = torch.where(amb, u - l, torch.ones_like(u))
        up = torch.where(amb, u / den, on)
        low = torch.where(amb, (u >= -l).double(), on) if crown else up
        return low, up, torch.where(amb, -l * u / den, torch.zeros_like(u))

    def crown(self, lo, up):
        """The CROWN duals and multipliers per layer."""
        lo, up = self.cut(lo), self.cut(up)
        lam, rho, lams = -self.W[-1].expand(lo[0].shape[0], -1), [None] * (self.n - 1), [None] * (self.n - 1)
        for k in range(self.n - 2, -1, -1):
            low, high, _ = self.relaxation(lo[k], up[k], True)
            lams[k], rho[k] = lam, high * lam.clamp(min=0) + low * lam.clamp(max=0)
            if k:
                lam = self.tr(k, rho[k])
        return rho, lams

    @staticmethod
    def vertex(r, g, l, u):
        """Minimiser of r x_hat - g x over the ReLU's hull: (x_hat, x, code)."""
        blk, pas = u <= 0, (l >= 0) & (u > 0)
        zero = torch.zeros_like(r)
        mag = TIE * (r.abs() + g.abs())
        code = torch.where(zero < r * l, 1, 0)
        best = torch.minimum(r * l, zero)
        code = torch.where((r - g) * u < best - mag * torch.maximum(-l, u), 2, code)
        code = torch.where(pas, torch.where(r - g <= mag, 2, 0), code)
        code = torch.where(blk, torch.where(r <= 0, 2, 0), code)
        xh = torch.where(code == 0, l, torch.where(code == 1, zero, u))
        x = torch.where(blk, zero, torch.where(pas, xh, torch.where(code == 2, u, zero)))
        return xh, x, code

    def inner(self, rho, l0, u0, lo, up):
        """Per layer g_k, x_k (from the input on) and x_hat_k, codes of the hidden layers."""
        top = -self.W[-1].expand(rho[0].shape[0], -1)
        g = [self.tr(k, rho[k]) for k in range(self.n - 1)] + [top]
        x, xh, code = [torch.where(g[0] >= 0, u0, l0)], [], []
        for k in range(self.n - 1):
            h, y, c = self.vertex(rho[k], g[k + 1], lo[k], up[k])
            x.append(y)
            xh.append(h)
            code.append(c)
        return g, x, xh, code

    def forward(self, k, x):
        return self.lin(k, x) + self.bias[k]

    def dual(self, rho, l0, u0, lo, up):
        g = [self.tr(k, rho[k]) for k in range(self.n - 1)] + [-self.W[-1].expand(rho[0].shape[0], -1)]
        q = torch.minimum(-g[0] * l0, -g[0] * u0).sum(1) + self.b[-1]
        for k in range(self.n - 1):
            r, c, l, u = rho[k], g[k + 1], lo[k], up[k]
            blk, pas = torch.minimum(r * l, r * u), torch.minimum((r - c) * l, (r - c) * u)
            amb = torch.minimum((r * l).clamp(max=0), (r - c) * u)
            q = q + torch.where(u <= 0, blk, torch.where(l >= 0, pas, amb)).sum(1) - r @ self.bias[k]
        return q

    def adam(self, l0, u0, lo, up, T):
        lo_, up_ = self.cut(lo), self.cut(up)
        rho = self.crown(lo, up)[0]
        m, v = [torch.zeros_like(r) for r in rho], [torch.zeros_like(r) for r in rho]
        for t in range(T):
            alpha = 1e-2 + (1e-4 - 1e-2) * t / max(T - 1, 1)
            _, x, xh, _ = self.inner(rho, l0, u0, lo_, up_)
            for k in range(self.n - 1):
                s = xh[k] - self.forward(k, x[k])
                m[k], v[k] = 0.9 * m[k] + 0.1 * s, 0.999 * v[k] + 0.001 * s * s
                rho[k] = rho[k] + alpha * (m[k] / (1 - 0.9 ** (t + 1))) / ((v[k] / (1 - 0.999 ** (t + 1))).sqrt() + 1e-8)
        return self.dual(rho, l0, u0, lo_, up_), rho

    def proximal(self, l0, u0, lo, up, T):
        """Method of multipliers: J block-coordinate Frank-Wolfe sweeps per iteration, momentum."""
        n, lo_, up_ = self.n, self.cut(lo), self.cut(up)
        eta0, eta1, mom, sweeps = ETA
        lam = self.crown(lo, up)[0]
        _, x, xB, _ = self.inner(lam, l0, u0, lo_, up_)
        xA = [self.forward(k, x[k]) for k in range(n)]
        pi = [torch.zeros_like(r) for r in lam]
        top = -torch.ones((l0.shape[0], 1), dtype=torch.float64, device="cuda")
        for t in range(T):
            eta = eta0 + (eta1 - eta0) * t / max(T - 1, 1)
            for _ in range(sweeps):
                for k in range(n):       # block (x_hat_B,k, x_hat_A,k+1), 0 = the input
                    lp = lam[k - 1] + (xB[k - 1] - xA[k - 1]) / eta if k else None
                    lq = lam[k] + (xB[k] - xA[k]) / eta if k < n - 1 else top
                    g = self.tr(k, lq)
                    if k:
                        zB, xk, _ = self.vertex(lp, g, lo_[k - 1], up_[k - 1])
                    else:
                        xk = torch.where(g >= 0, u0, l0)
                    dA = self.forward(k, xk) - xA[k]
                    num, den = (lq * dA).sum(1), (dA * dA).sum(1) / eta if k < n - 1 else torch.zeros_like(top[:, 0])
                    if k:
                        dB = zB - xB[k - 1]
                        num, den = num - (lp * dB).sum(1), den + (dB * dB).sum(1) / eta
                    step = torch.where(den > 0, (num / torch.where(den > 0, den, 1.0)).clamp(0, 1), (num > 0).double())
                    if k:
                        xB[k - 1] = xB[k - 1] + step[:, None] * dB
                    xA[k] = xA[k] + step[:, None] * dA
            for k in range(n - 1):
                pi[k] = mom * pi[k] + (xB[k] - xA[k]) / eta
                lam[k] = lam[k] + pi[k]
        return self.dual(lam, l0, u0, lo_, up_), lam

    def substitute(self, k, rows, l0, u0, lo, up, crown):
        """Lower bounds of rows^T x_hat_k (k from 0) over one box per row; lo, up: bounds of the layers before."""
        val, a = rows @ self.bias[k], self.tr(k, rows)
        for j in range(k - 1, -1, -1):
            low, high, icp = self.relaxation(lo[j], up[j], crown)
            pos, neg = a.clamp(min=0), a.clamp(max=0)
            mu = low * pos + high * neg
            val = val + (neg * icp).sum(1) + mu @ self.bias[j]
            a = self.tr(j, mu)
        return val + torch.minimum(a * l0, a * u0).sum(1)

    def propagated(self, l0, u0, mask):
        """Layer-wise best of CROWN and WK for one box [1, n0] and its split mask."""
        los, ups = [], []
        for k in range(self.n - 1):
            eye = torch.eye(self.width[k], dtype=torch.float64, device="cuda")
            lo = up = None
            for crown in (True, False):
                a = torch.cat([self.substitute(k, e, l0, u0, los, ups, crown) for e in eye.split(512)])
                b = -torch.cat([self.substitute(k, -e, l0, u0, los, ups, crown) for e in eye.split(512)])
                lo, up = (a, b) if lo is None else (torch.maximum(lo, a), torch.minimum(up, b))
            if mask is not None:
                m = self.cut(mask)[k][0]
                lo, up = torch.where(m > 0, lo.clamp(min=0), lo), torch.where(m < 0, up.clamp(max=0), up)
            los.append(lo[None])
            ups.append(up[None])
        return torch.cat(los, 1), torch.cat(ups, 1)


def exact(case, seed):
    i = _Inputs(case, seed)
    net, kind = i.ref, case["kind"]
    with torch.no_grad():
        if kind in ("bound", "proximal"):
            l0, u0 = i.boxes()
            lo, up = i.clamped()
            solve = net.adam if kind == "bound" else net.proximal
            parts = [solve(*(t[b : b + 512] for t in (l0, u0, lo, up)), case["T"]) for b in range(0, case["B"], 512)]
            return {"bound": torch.cat([q for q, _ in parts]), "rho": torch.cat([torch.cat(r, 1) for _, r in parts])}
        if kind == "grad":
            l0, u0 = i.boxes()
            q, _ = net.adam(l0, u0, *i.clamped(), case["T"])
            # the gradients are those of the iterate's own vertex choices, which rounding decides: no 64-bit value
            return {"bound": q, "grads": None}
        if kind == "interval":
            lo, up, out = net.interval(i.l0.double(), i.u0.double(), output=True)
            return {"lower": lo, "upper": up, "output": out}
        if kind == "propagated":
            rows = case["B"] or case["P"]
            got = []
            for r in range(rows):
                p = r if not case["B"] else 0 if i.prop is None else int(i.prop[r])
                m = i.masks[r : r + 1] if i.masks is not None else None
                got.append(net.propagated(i.l0[p : p + 1].double(), i.u0[p : p + 1].double(), m))
            return {"lower": torch.cat([g[0] for g in got]), "upper": torch.cat([g[1] for g in got])}
        if kind == "fsb":
            return {"decision": None, "children": _children(i)}
        l0, u0 = i.boxes()
        lo, up = (net.cut(t) for t in i.clamped())
        rho = net.cut(i.rho.double())
        _, x, xh, code = net.inner(rho, l0, u0, lo, up)
        sg = [xh[k] - net.forward(k, x[k]) for k in range(net.n - 1)]
        y = x[0]
        for k in range(net.n):
            y = net.forward(k, y).clamp(min=0) if k < net.n - 1 else net.forward(k, y)
        return {"q": net.dual(rho, l0, u0, lo, up), "supergradient": torch.cat(sg, 1), "vertex": None,
                "upper": y[:, 0], "x0": x[0]}


def _children(i):
    """Output bounds of the children of every layer's two branching candidates [B, candidates, 2]."""
    net = i.ref
    l0, u0 = i.boxes()
    lo, up = i.clamped()
    los, ups = net.cut(lo), net.cut(up)
    lam, cand, off = -net.W[-1].expand(lo.shape[0], -1), [None] * (net.n - 1), np.cumsum([0, *net.width])
    for k in range(net.n - 2, -1, -1):
        l, u = los[k], ups[k]
        amb = (l < 0) & (u > 0)
        slope = torch.where(amb, u / torch.where(amb, u - l, torch.ones_like(u)), (u > 0).double())
        icp = torch.where(amb, u * l / torch.where(amb, u - l, torch.ones_like(u)), torch.zeros_like(u)) * lam.clamp(min=0)
        lb = lam * net.bias[k]
        score = (lb.clamp(max=0) - slope * lb + icp).abs()
        none = torch.full_like(l, -math.inf)
        cand[k] = [int(off[k]) + torch.where(amb, s, none).argmax(1) for s in (score, -icp)]
        if k:
            lam = net.tr(k, slope * lam)
    row = torch.arange(lo.shape[0], device="cuda")
    one = torch.ones((lo.shape[0], 1), dtype=torch.float64, device="cuda")
    out = []
    for c in (c for pair in cand for c in pair):
        l2, u2 = lo.clone(), up.clone()
        l2[row, c], u2[row, c] = l2[row, c].clamp(min=0), u2[row, c].clamp(max=0)
        both = [torch.maximum(*(net.substitute(net.n - 1, one, l0, u0, net.cut(l), net.cut(u), r) for r in (True, False)))
                for l, u in ((l2, up), (lo, u2))]
        out.append(torch.stack(both, 1))
    return torch.stack(out, 1)
