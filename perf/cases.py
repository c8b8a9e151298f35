"""The work that programs have this library do, as a list of cases and a generator of more of the same ranges.

A case names one call sequence through the public entry points (`op`), a network (`widths`), the number of training
rows (`l`) and of subsampled rows (`nS`), the distribution of the features (`x`) and the precision mode of the context
(`prec`), plus what the call itself takes.  The operations:

    gv       one product G^S v (what a solver of the caller's own asks for)
    block    one block-diagonal product Ghat^S v, with `split` for a partition of the variables finer than layers
    cg       a conjugate-gradient solve of `steps` steps on the full system, or (`blockdiag`) the block systems; the
             block solve starts from a fresh subsample, as it does in every Newton iteration
    first    the first product on a new subsample: row gather, stored forward pass, G^S v
    grad     f and its gradient over all rows
    fun      f over all rows (one trial point of a line search)
    newton   one whole Newton iteration: gradient, block CG, combination of directions, line search
"""
import math

import numpy as np
import torch

import paper_1802_00130_b200 as gn

DEVICE = "cuda:0"
LAMBDA = 1.0            # the Levenberg-Marquardt term a solve starts with


def _case(name, op, widths, nS, l, x, prec, **more):
    return dict(name=name, op=op, widths="-".join(str(w) for w in widths), nS=nS, l=l, x=x, prec=prec, **more)


def listed():
    return [
        # the smallest network: nothing but launches and latency
        _case("gv_tiny", "gv", [20, 16, 16, 4], 64, 256, "uniform", "fp32"),
        # small, every width odd: the gradient of a toy problem or of one mini-batch
        _case("grad_ragged", "grad", [37, 53, 19, 7], 131, 333, "sparse80", "fp32"),
        # two-class, scalar output; the solver looks at its stop rule after every step (the tolerance is not reached)
        _case("cg_binary300", "cg", [28, 300, 300, 1], 2000, 20000, "normal", "fp32", steps=10, tol=1e-3),
        # an ordinary small image network, 5 % subsample: one product
        _case("gv_mnist300", "gv", [784, 300, 300, 10], 3000, 60000, "sparse80", "tf32"),
        # ... and one whole Newton iteration on it in the default precision
        _case("newton_mnist300", "newton", [784, 300, 300, 10], 3000, 60000, "sparse80", "fp32", steps=10),
        # dense features, a fixed number of CG steps on the full system
        _case("cg_svhn1000", "cg", [3072, 1000, 1000, 10], 2500, 50000, "uniform", "fp32", steps=20, tol=0.0),
        # widths as a feature selection leaves them (no multiple of four), more than 16 classes
        _case("block_odd", "block", [617, 1201, 803, 26], 4001, 8002, "normal", "tf32"),
        # a split variable partition (12 blocks instead of 4)
        _case("split_mnist2000", "block", [784, 2000, 2000, 2000, 10], 3000, 60000, "sparse80", "tf32", split="1-2-2-2-1"),
        # the block-diagonal solve of a Newton iteration at the large image network, 20 % subsample
        _case("blockcg_mnist2000", "cg", [784, 2000, 2000, 2000, 10], 12000, 60000, "sparse80", "tf32", steps=10, tol=0.0,
              blockdiag=True),
        # one product there, in both precisions
        _case("gv_mnist2000", "gv", [784, 2000, 2000, 2000, 10], 12000, 60000, "sparse80", "tf32"),
        _case("gv_mnist2000_fp32", "gv", [784, 2000, 2000, 2000, 10], 12000, 60000, "sparse80", "fp32"),
        # the largest: gradient over all rows of a wide, deep network
        _case("grad_wide4096", "grad", [1024, 4096, 4096, 4096, 4096, 100], 20000, 200000, "normal", "tf32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any operation, one to five layers, round and odd widths, 64 to 60000 subsampled rows."""
    while True:
        op = rng.choice(["gv", "gv", "gv", "block", "block", "cg", "cg", "first", "grad", "grad", "fun", "newton"])
        L = rng.choice([1, 2, 3, 3, 4, 5])
        widths = [_log_int(rng, 16, 3072)] + [_log_int(rng, 16, 4096) for _ in range(L - 1)] + [_log_int(rng, 1, 100)]
        if rng.random() < 0.6:                                      # round hidden widths
            widths = [w if m in (0, L) else (w + 49) // 50 * 50 for m, w in enumerate(widths)]
        if rng.random() < 0.5:
            widths[0] = (widths[0] + 3) // 4 * 4
        nS = _log_int(rng, 64, 60000)
        l = min(200000, nS * rng.choice([1, 2, 5, 10, 20]))
        prec = rng.choice(["tf32", "fp32"])
        case = dict(op=op, widths="-".join(str(w) for w in widths), nS=nS, l=l, x=rng.choice(["sparse80", "uniform", "normal"]),
                    prec=prec)
        # (the narrowest systems have 17 unknowns: they stay short of the step at which their residual is exactly zero)
        if op == "cg":
            case.update(steps=rng.randint(3, 8), tol=0.0, blockdiag=rng.random() < 0.5)
        if op == "newton":
            case.update(steps=rng.randint(3, 8))
        if op == "block" and L >= 2 and widths[-1] <= 32 and rng.random() < 0.3:
            case.update(split="-".join(str(1 if m in (0, L) else rng.randint(1, min(4, w))) for m, w in enumerate(widths)))
        most = work(listed()[-1])["flops"]
        if prec == "fp32":
            most /= 4
        factors = 4 * nS * widths[-1] * sum(widths[1:-1]) if widths[-1] <= 32 else 0
        if work(case)["flops"] <= most / 2 and factors <= 6e9 and l * widths[0] <= 2.5e8 and L * nS * sum(widths) <= 2.5e9:
            return case


def _widths(case):
    return [int(w) for w in case["widths"].split("-")]


def _features(kind, rows, cols, g):
    if kind == "normal":
        return torch.randn(rows, cols, device=DEVICE, generator=g)
    x = torch.rand(rows, cols, device=DEVICE, generator=g)
    if kind == "sparse80":                                          # mostly-zero pixels
        x *= torch.rand(rows, cols, device=DEVICE, generator=g) < 0.2
    return x


def _inputs(case, seed):
    widths, l, nS = _widths(case), case["l"], case["nS"]
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    X = _features(case["x"], l, widths[0], g)
    if widths[-1] == 1:                                             # two classes: labels -1 / +1
        Y = (2.0 * torch.randint(0, 2, (l, 1), device=DEVICE, generator=g) - 1.0).float()
    else:
        labels = torch.randint(0, widths[-1], (l,), device=DEVICE, generator=g)
        Y = torch.zeros(l, widths[-1], device=DEVICE)
        Y[torch.arange(l, device=DEVICE), labels] = 1.0
    parts = []
    for a, b in zip(widths[:-1], widths[1:]):                       # W^m, b^m ~ N(0, 1 / fan-in)
        parts.append(torch.randn((a + 1) * b, device=DEVICE, generator=g) / math.sqrt(a))
    theta = torch.cat(parts)
    idx = torch.randperm(l, device=DEVICE, generator=g)[:nS].to(torch.int32)
    v = torch.randn(theta.numel(), device=DEVICE, generator=g)
    return X, Y, theta, idx, v


def prepare(case, seed):
    widths, l, op = _widths(case), case["l"], case["op"]
    X, Y, theta, idx, v = _inputs(case, seed)
    ctx = gn.GnContext(widths, float(l), X, Y, gn.GN_TF32 if case["prec"] == "tf32" else gn.GN_FP32_ACCURATE)
    if case.get("split"):
        ctx.set_split([int(s) for s in case["split"].split("-")])
    s = dict(case=case, ctx=ctx, theta=theta, idx=idx, v=v, out=torch.empty_like(theta))
    if op == "newton":
        s.update(theta_new=torch.empty_like(theta), direction=torch.empty_like(theta),
                 params=gn.NewtonParams(lam=LAMBDA, sigma=0.0, cg_max=case["steps"], blockdiag=1))
        return s
    ctx.set_theta(theta)
    if op in ("gv", "block", "cg"):
        ctx.set_subsample(idx)
    if op == "cg":
        s["g"] = ctx.grad()                                         # the right-hand side of a solve
    return s


def run(s):
    case, ctx = s["case"], s["ctx"]
    op = case["op"]
    if op == "gv":
        return ctx.Gv(s["v"], out=s["out"])
    if op == "block":
        return ctx.Gv_blockdiag(s["v"], out=s["out"])
    if op == "cg":
        block = bool(case.get("blockdiag"))
        if block:
            ctx.set_subsample(s["idx"])
        d, steps, res = ctx.cg_solve(s["g"], LAMBDA, blockdiag=block, max_iter=case["steps"], tol=case["tol"], out=s["out"])
        return {"d": d, "steps": steps, "residuals": np.asarray(res)}
    if op == "first":
        ctx.set_subsample(s["idx"])
        return ctx.Gv(s["v"], out=s["out"])
    if op == "grad":
        g, f = ctx.grad(out=s["out"], with_f=True)
        return {"g": g, "f": f}
    if op == "fun":
        return ctx.fun()
    s["theta_new"].copy_(s["theta"])                                # both are updated in place
    s["direction"].zero_()
    rep = ctx.newton_iter(s["theta_new"], s["idx"], s["direction"], s["params"])
    return {"theta": s["theta_new"], "direction": s["direction"], "f_before": rep["f_before"], "f_after": rep["f_after"]}


class _Exact:
    """The same mathematics in 64 bits: explicit layers, rows taken `ROWS` at a time."""
    ROWS = 16384

    def __init__(self, case, seed):
        X, Y, theta, idx, v = _inputs(case, seed)
        self.widths, self.l, self.X, self.Y, self.S = _widths(case), case["l"], X, Y, idx.long()
        self.theta, self.v, self.C = theta.double(), v.double(), float(case["l"])
        self.L = len(self.widths) - 1
        self.masks = self._masks([int(s) for s in case["split"].split("-")]) if case.get("split") else None

    def layers(self, vec):
        """[(W^m as n_m x n_{m-1}, b^m)] views of a vector laid out like theta."""
        out, at = [], 0
        for a, b in zip(self.widths[:-1], self.widths[1:]):
            out.append((vec[at:at + a * b].view(b, a), vec[at + a * b:at + (a + 1) * b]))
            at += (a + 1) * b
        return out

    def _masks(self, split):
        """One vector of booleans per partition: group a of layer m - 1 to group b of layer m, biases with a = 0."""
        group = [torch.zeros(w, dtype=torch.long, device=DEVICE) for w in self.widths]
        for w, s, gr in zip(self.widths, split, group):
            for k in range(s):
                gr[k * w // s:(k + 1) * w // s] = k
        masks = []
        for m in range(1, self.L + 1):
            for a in range(split[m - 1]):
                for b in range(split[m]):
                    mask = torch.zeros_like(self.theta, dtype=torch.bool)
                    W, bias = self.layers(mask)[m - 1]
                    W.copy_((group[m] == b)[:, None] & (group[m - 1] == a)[None, :])
                    bias.copy_((group[m] == b) & (a == 0))
                    masks.append(mask)
        return masks

    def forward(self, theta, x):
        z = [x.double()]
        for m, (W, b) in enumerate(self.layers(theta), 1):
            s = torch.addmm(b, z[-1], W.T)
            z.append(torch.sigmoid(s) if m < self.L else s)
        return z

    def backward(self, z, delta, out, scale, lowest=1):
        """out += scale J^T delta for the layers from `lowest` up."""
        W, O = self.layers(self.theta_now), self.layers(out)
        for m in range(self.L, lowest - 1, -1):
            O[m - 1][0].addmm_(delta.T, z[m - 1], alpha=scale)
            O[m - 1][1].add_(delta.sum(0), alpha=scale)
            if m > lowest:
                delta = (delta @ W[m - 1][0]) * z[m - 1] * (1 - z[m - 1])

    def fun(self, theta, grad=None):
        self.theta_now, loss = theta, 0.0
        for r in range(0, self.l, self.ROWS):
            z = self.forward(theta, self.X[r:r + self.ROWS])
            d = z[-1] - self.Y[r:r + self.ROWS]
            loss += float((d * d).sum())
            if grad is not None:
                self.backward(z, 2 * d, grad, 1.0 / self.l)
        if grad is not None:
            grad.add_(theta, alpha=1.0 / self.C)
        return float(theta @ theta) / (2 * self.C) + loss / self.l

    def grad(self):
        g = torch.zeros_like(self.theta)
        f = self.fun(self.theta, g)
        return g, f

    def Gv(self, v, blocks=False):
        """G^S v, or, `blocks`, the part of it that stays inside each block (layer, or partition of the split)."""
        self.theta_now, out = self.theta, v / self.C
        W, n = self.layers(self.theta), self.S.numel()
        if not blocks:
            parts = [None]
        elif self.masks is None:
            parts = list(range(1, self.L + 1))
        else:
            parts = self.masks
        for r in range(0, n, self.ROWS):
            z = self.forward(self.theta, self.X[self.S[r:r + self.ROWS]])
            for part in parts:
                mask = part if torch.is_tensor(part) else None
                V = self.layers(v if mask is None else v * mask)
                only = range(1, self.L + 1) if not isinstance(part, int) else [part]
                rz = torch.zeros_like(z[0])
                for m in range(1, self.L + 1):
                    rs = rz @ W[m - 1][0].T
                    if m in only:
                        rs += torch.addmm(V[m - 1][1], z[m - 1], V[m - 1][0].T)
                    rz = rs * z[m] * (1 - z[m]) if m < self.L else rs
                if part is None:
                    self.backward(z, 2 * rz, out, 1.0 / n)
                    continue
                add = torch.zeros_like(out)
                if isinstance(part, int):
                    self.backward(z, 2 * rz, add, 1.0 / n, part)
                    for m, (A, b) in enumerate(self.layers(add), 1):
                        if m != part:
                            A.zero_(), b.zero_()
                else:
                    self.backward(z, 2 * rz, add, 1.0 / n)
                    add *= mask
                out += add
        return out

    def cg(self, g, steps, blocks, tol=0.0):
        """At most `steps` steps of conjugate gradient from zero; one independent solve per layer with `blocks`."""
        ends = [0]
        for a, b in zip(self.widths[:-1], self.widths[1:]):
            ends.append(ends[-1] + (a + 1) * b)
        spans = [slice(a, b) for a, b in zip(ends[:-1], ends[1:])] if blocks else [slice(0, ends[-1])]
        d, r = torch.zeros_like(g), -g
        p, rho = r.clone(), [float(r[s] @ r[s]) for s in spans]
        norms, goal = [math.sqrt(sum(rho))], [tol * math.sqrt(k) for k in rho]
        for _ in range(steps):
            if all(math.sqrt(k) <= t for k, t in zip(rho, goal)):
                break
            q = self.Gv(p, blocks) + LAMBDA * p
            for k, s in enumerate(spans):
                pq = float(p[s] @ q[s])
                if math.sqrt(rho[k]) <= goal[k]:
                    continue                # this solve has met its test
                alpha = rho[k] / pq
                d[s] += alpha * p[s]
                r[s] -= alpha * q[s]
                new = float(r[s] @ r[s])
                p[s] = r[s] + new / rho[k] * p[s]
                rho[k] = new
            norms.append(math.sqrt(sum(rho)))
        return d, norms

    def newton(self, steps):
        eta, max_backtrack = 1e-4, 30       # what NewtonParams sets where a caller does not
        g, f0 = self.grad()
        d, _ = self.cg(g, steps, True)      # (the previous direction is zero: the two-variable system reduces to d)
        alpha, slope, f1 = 1.0, float(g @ d), 0.0
        for k in range(max_backtrack + 1):
            f1 = self.fun(self.theta + alpha * d)
            if f1 <= f0 + eta * alpha * slope or k == max_backtrack:
                break
            alpha /= 2
        return {"theta": self.theta + alpha * d, "direction": d, "f_before": f0, "f_after": f1}


def exact(case, seed):
    op = case["op"]
    if case.get("split"):
        s = [int(k) for k in case["split"].split("-")]
        if sum(a * b for a, b in zip(s[:-1], s[1:])) * _macs(_widths(case))["gv"] * 2.0 * case["nS"] > 1.5e14:
            return None                     # (one pass per partition)
    e = _Exact(case, seed)
    if op in ("gv", "first"):
        return e.Gv(e.v)
    if op == "block":
        return e.Gv(e.v, True)
    if op == "cg":
        d, norms = e.cg(e.grad()[0], case["steps"], bool(case.get("blockdiag")), case["tol"])
        return {"d": d, "steps": None, "residuals": np.asarray(norms)}
    if op == "grad":
        g, f = e.grad()
        return {"g": g, "f": f}
    if op == "fun":
        return e.fun(e.theta)
    return e.newton(case["steps"])


def _macs(widths):
    """Multiply-adds per row: forward pass, gradient, full product, block product (through the n_L x n_m factors)."""
    g = [a * b for a, b in zip(widths[:-1], widths[1:])]
    return dict(fun=sum(g), grad=3 * sum(g) - g[0], gv=4 * sum(g) - 2 * g[0],
                block=2 * sum(g) + 2 * widths[-1] * sum(widths[1:]))


def work(case):
    widths, l, nS, op = _widths(case), case["l"], case["nS"], case["op"]
    mac = _macs(widths)
    n = sum((a + 1) * b for a, b in zip(widths[:-1], widths[1:]))
    acts, data = 4.0 * nS * sum(widths), 4.0 * l * (widths[0] + widths[-1])
    product = lambda kind: (2.0 * nS * mac[kind], acts + 12.0 * n)  # activations, theta and v in, the product out
    if op in ("gv", "block"):
        flops, nbytes = product(op)
    elif op == "first":
        flops, nbytes = 2.0 * nS * (mac["fun"] + mac["gv"]), acts + 4.0 * nS * widths[0] + 12.0 * n
    elif op in ("fun", "grad"):
        flops, nbytes = 2.0 * l * mac[op], data + 4.0 * n * (2 if op == "grad" else 1)
    elif op == "cg":
        f, b = product("block" if case.get("blockdiag") else "gv")
        flops, nbytes = case["steps"] * f, case["steps"] * b
        if case.get("blockdiag"):
            flops, nbytes = flops + 2.0 * nS * mac["fun"], nbytes + acts
    else:                                                           # newton: subsample, gradient, solve, two products, one trial f
        (fb, bb), (ff, bf) = product("block"), product("gv")
        flops = 2.0 * nS * mac["fun"] + 2.0 * l * (mac["grad"] + mac["fun"]) + case["steps"] * fb + 2 * ff
        nbytes = acts + 2 * data + case["steps"] * bb + 2 * bf + 16.0 * n
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # Four times the largest difference seen between this path and the same calls with every contraction summed in
    # another order in 32 bits.  A solve multiplies the rounding of its products by the condition of its system.
    solve = case["op"] in ("cg", "newton")
    if case["prec"] == "fp32":
        return {"rel": 1.6e-3 if solve else 5e-6}
    return {"rel": 1.5e-2 if solve else 2e-3}
