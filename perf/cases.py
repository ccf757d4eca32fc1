"""What is timed: calls of the library's public entry points, over the sizes its users run.

A user of this library fits an occupancy field, pushes planner samples through
the diffeomorphism, differentiates it, scores samples under it, does so for
many environments at once, and trains and runs the surrogate network.  The
listed cases follow that life; their sizes are the repository's own workloads
(the 2-D grid field, the 2-D fitted field, the 7-D random Fourier field, the
batched environments, the 3-D surrogate), scaled to one planner call where the
workload itself is a stress size, with odd and ragged counts among them.

Inputs are drawn on the GPU from the seed alone, nothing on the way to them
uses the library.  The step size of a map is 0.05 over a sampled bound of the
cost's Hessian: between the certified step (0.5 over a bound some ten to a
thousand times the sampled one) and the largest that keeps a chain a
diffeomorphism, so that samples move visibly and the map stays as well
conditioned as a planner's.
"""
import math

import torch

import paper_2108_11775_gb300 as pdmp

RBF, RFF = "rbf", "rff"


# ------------------------------------------------------------------- the cases
def listed():
    return [
        # one planner query on a small map: the smallest call, launches and latency count
        {"name": "morph-grid", "op": "morph", "kind": RBF, "d": 2, "M": 1024, "N": 4096, "T": 10, "gamma": 4.0,
         "side": 10.0, "layout": "grid", "weights": "normal"},
        # a fitted 2-D map at scale: the headline workload, the largest call
        {"name": "morph-fitted", "op": "morph", "kind": RBF, "d": 2, "M": 16384, "N": 1 << 20, "T": 50, "gamma": 8.0,
         "side": 10.0, "weights": "fitted"},
        # a batch of 7-D arm configurations through a random Fourier field
        {"name": "morph-arm", "op": "morph", "kind": RFF, "d": 7, "M": 4096, "N": 20000, "T": 20, "weights": "normal"},
        # training through the map (forward with checkpoints, then gradients to samples, weights and bias)
        {"name": "grad-arm", "op": "grad", "kind": RFF, "d": 7, "M": 4096, "N": 65537, "T": 20, "k": 5,
         "weights": "normal"},
        {"name": "grad-fitted", "op": "grad", "kind": RBF, "d": 2, "M": 8192, "N": 30011, "T": 50, "k": 5, "gamma": 8.0,
         "side": 10.0, "weights": "fitted"},
        # the volume change of the map, for density work in 7-D
        {"name": "logdet-arm", "op": "logdet", "kind": RFF, "d": 7, "M": 4096, "N": 131072, "T": 20,
         "weights": "normal"},
        # scoring samples: the inverse map and its log-density
        {"name": "density-fitted", "op": "density", "kind": RBF, "d": 2, "M": 16384, "N": 65536, "T": 50, "gamma": 8.0,
         "side": 10.0, "weights": "fitted"},
        # many planner instances in one launch, uneven sizes, 2-D and 3-D
        {"name": "batch-environments", "op": "batch", "envs": 48, "M_lo": 256, "M_hi": 8192, "N_lo": 1024,
         "N_hi": 65536, "T": 30},
        # the surrogate network: inference on a sampler's bucket, and one training step
        {"name": "surrogate-forward", "op": "forward", "N": 4194304},
        {"name": "surrogate-train", "op": "train", "B": 4096},
        # fitting the occupancy map to labelled points
        {"name": "fit-map", "op": "fit", "d": 2, "M": 4096, "n": 50000, "gamma": 8.0, "side": 10.0, "power": 20,
         "iters": 60},
        # collision queries on the fitted map: c, s and grad c at the points of a roadmap's edges
        {"name": "query-edges", "op": "query", "kind": RBF, "d": 2, "M": 16384, "N": 100003, "gamma": 8.0, "side": 10.0,
         "weights": "fitted"},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _rbf_shape(rng):
    d = rng.choice((2, 2, 3))
    return {"kind": RBF, "d": d, "gamma": rng.choice((4.0, 8.0)), "side": 10.0 if d == 2 else rng.choice((5.0, 10.0)),
            "weights": rng.choice(("normal", "fitted"))}


def draw(rng):
    op = rng.choice(("morph", "morph", "morph", "grad", "grad", "logdet", "density", "batch", "forward", "train", "fit",
                     "query"))
    if op == "morph":
        if rng.random() < 0.6:
            c = {"op": op, **_rbf_shape(rng), "M": _log_int(rng, 256, 16384), "T": rng.randint(10, 50)}
            top = min(1 << 20, int(4e11 / (c["M"] * c["T"])))
        else:
            c = {"op": op, "kind": RFF, "d": rng.randint(2, 7), "M": _log_int(rng, 512, 4096), "T": rng.randint(10, 20),
                 "weights": "normal"}
            top = min(1 << 20, int(8e10 / (c["M"] * c["T"])))
        c["N"] = _log_int(rng, 1024, max(1024, top))
    elif op == "grad":
        k = rng.choice((2, 5))
        if rng.random() < 0.5:
            c = {"op": op, **_rbf_shape(rng), "M": _log_int(rng, 256, 16384), "T": k * rng.randint(2, 10), "k": k}
            top = min(1 << 18, int(1e11 / (c["M"] * c["T"])))
        else:
            c = {"op": op, "kind": RFF, "d": rng.randint(2, 7), "M": _log_int(rng, 512, 4096), "T": k * rng.randint(2, 4),
                 "k": k, "weights": "normal"}
            top = min(1 << 18, int(2e10 / (c["M"] * c["T"])))
        c["N"] = _log_int(rng, 1024, max(1024, top))
    elif op == "logdet":
        c = {"op": op, "kind": RFF, "d": rng.randint(2, 7), "M": _log_int(rng, 512, 4096), "T": rng.randint(10, 20),
             "weights": "normal"}
        c["N"] = _log_int(rng, 1024, max(1024, min(1 << 18, int(2e10 / (c["M"] * c["T"])))))
    elif op == "density":
        c = {"op": op, **_rbf_shape(rng), "M": _log_int(rng, 256, 16384), "T": rng.randint(10, 50)}
        c["N"] = _log_int(rng, 1024, max(1024, min(1 << 18, int(6e10 / (c["M"] * c["T"])))))
    elif op == "batch":
        c = {"op": op, "envs": rng.randint(4, 48), "M_lo": 256, "M_hi": _log_int(rng, 1024, 8192), "N_lo": 1024,
             "N_hi": _log_int(rng, 4096, 65536), "T": rng.randint(10, 30)}
    elif op == "forward":
        c = {"op": op, "N": _log_int(rng, 1024, 1 << 24)}
    elif op == "train":
        c = {"op": op, "B": _log_int(rng, 256, 16384)}
    elif op == "fit":
        d = rng.choice((2, 2, 3))
        c = {"op": op, "d": d, "M": _log_int(rng, 256, 8192), "n": _log_int(rng, 5000, 100000), "gamma": 8.0,
             "side": 10.0 if d == 2 else 5.0, "power": 20, "iters": rng.randint(30, 100)}
    else:
        kind = rng.choice((RBF, RBF, RFF))
        if kind == RBF:
            c = {"op": op, **_rbf_shape(rng), "M": _log_int(rng, 256, 16384)}
        else:
            c = {"op": op, "kind": RFF, "d": rng.randint(2, 7), "M": _log_int(rng, 512, 4096), "weights": "normal"}
        c["N"] = _log_int(rng, 1000, 1 << 20)
    return c


# ------------------------------------------------------------------- the inputs
class _Draws:
    """Seeded draws on the GPU."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed))

    def uniform(self, shape, lo, hi):
        return torch.rand(shape, generator=self.g, device="cuda", dtype=torch.float32) * (hi - lo) + lo

    def normal(self, *shape):
        return torch.randn(shape, generator=self.g, device="cuda", dtype=torch.float32)


def _boxes(r, nb, d, side):
    c = r.uniform((nb, d), 0.0, side)
    h = 0.5 * r.uniform((nb, d), 0.03 * side, 0.15 * side)
    return c - h, c + h


def _inside(lo, hi, x):
    y = torch.zeros(x.shape[0], dtype=torch.bool, device="cuda")
    for a, b in zip(lo, hi):
        y |= ((a <= x) & (x <= b)).all(dim=1)
    return y


def _field(r, c):
    """{kind, centres, w, gamma, phase, bias} of a case's field."""
    d, M = c["d"], c["M"]
    if c["kind"] == RFF:
        return {"kind": RFF, "centres": math.sqrt(2.0) * r.normal(M, d), "phase": r.uniform((M,), 0.0, 2.0 * math.pi),
                "w": r.normal(M) / math.sqrt(M), "gamma": 0.0, "bias": 0.0}
    side = c["side"]
    if c.get("layout") == "grid":           # the 32 x 32 edge-inclusive grid
        g = torch.linspace(0.0, side, 32, device="cuda")
        mu = torch.stack(torch.meshgrid(g, g, indexing="ij"), dim=-1).reshape(-1, 2).contiguous()
    else:
        mu = r.uniform((M, d), 0.0, side)
    if c["weights"] == "normal":
        w, bias = r.normal(M), 0.0
    else:                                   # the signs and spread of a fitted map
        lo, hi = _boxes(r, 64, d, side)
        occ = _inside(lo, hi, mu).float()
        w, bias = 0.5 * (2.0 * occ - 1.0) * (0.5 + 0.5 * r.normal(M).abs()), -0.5
    return {"kind": RBF, "centres": mu, "phase": None, "w": w, "gamma": c["gamma"], "bias": bias}


def _box(c):
    return (-math.pi, math.pi) if c.get("kind") == RFF else (0.0, c["side"])


def _moments(f, x, hess=True):
    """s, grad s and Hess s at the rows of x in 64 bits (f: 64-bit tensors)."""
    mu, w = f["centres"], f["w"]
    if f["kind"] == RBF:
        gm = f["gamma"]
        r2 = torch.zeros(x.shape[0], mu.shape[0], dtype=x.dtype, device=x.device)
        for j in range(mu.shape[1]):
            r2 = r2 + (x[:, j:j + 1] - mu[:, j]) ** 2
        e = torch.exp(-gm * r2) * w
        S, m = e.sum(1), e @ mu
        g = -2.0 * gm * (x * S[:, None] - m)
        if not hess:
            return S + f["bias"], g, None
        mm = (e @ (mu[:, :, None] * mu[:, None, :]).reshape(mu.shape[0], -1)).reshape(x.shape[0], x.shape[1], -1)
        xm = x[:, :, None] * m[:, None, :]
        q = S[:, None, None] * (x[:, :, None] * x[:, None, :]) - xm - xm.transpose(1, 2) + mm
        eye = torch.eye(x.shape[1], dtype=x.dtype, device=x.device)
        return S + f["bias"], g, 4.0 * gm * gm * q - 2.0 * gm * S[:, None, None] * eye
    th = x @ mu.t() + f["phase"]
    cw = torch.cos(th) * w
    g = -(torch.sin(th) * w) @ mu
    if not hess:
        return cw.sum(1) + f["bias"], g, None
    H = -(cw @ (mu[:, :, None] * mu[:, None, :]).reshape(mu.shape[0], -1)).reshape(x.shape[0], x.shape[1], -1)
    return cw.sum(1) + f["bias"], g, H


def _double(f):
    return {k: v.double() if isinstance(v, torch.Tensor) else v for k, v in f.items()}


def _eta(f, lo, hi):
    """0.05 over the largest bound |Hess c| <= |Hess s| / 4 + |grad s|^2 / (6 sqrt 3) at 1024 fixed points."""
    r = _Draws(17)
    x = r.uniform((1024, f["centres"].shape[1]), lo, hi).double()
    _, g, H = _moments(_double(f), x)
    L = (torch.linalg.matrix_norm(H) / 4.0 + (g * g).sum(1) / (6.0 * math.sqrt(3.0))).max()
    return float((0.05 / L).float())


def _map(case, seed):
    """The field, the samples and the step size of a case that has one field."""
    r = _Draws(seed)
    f = _field(r, case)
    lo, hi = _box(case)
    return r, f, r.uniform((case["N"], case["d"]), lo, hi), _eta(f, lo, hi)


def _environments(case, seed):
    """A batch's environments: sizes from the case alone, contents from the seed."""
    import random
    sizes = random.Random(1000 * case["envs"] + case["T"])
    r, envs = _Draws(seed), []
    for _ in range(case["envs"]):
        d = sizes.choice((2, 3))
        M, N = sizes.randint(case["M_lo"], case["M_hi"]), sizes.randint(case["N_lo"], case["N_hi"])
        f = _field(r, {"kind": RBF, "d": d, "M": M, "gamma": 4.0, "side": 10.0, "weights": "normal"})
        envs.append((f, r.uniform((N, d), 0.0, 10.0), _eta(f, 0.0, 10.0)))
    return envs


def _pairs(r, n):
    """Training pairs in [0, 5]^3: points and a displacement field with the sharpness of a morph's."""
    x = r.uniform((n, 3), 0.0, 5.0)
    return x, x + 0.02 * torch.tanh(4.0 * torch.sin(2.5 * x.roll(1, 1)) * torch.cos(1.5 * x))


def _labelled(case, seed):
    r = _Draws(seed)
    mu = r.uniform((case["M"], case["d"]), 0.0, case["side"])
    lo, hi = _boxes(r, 64, case["d"], case["side"])
    X = r.uniform((case["n"], case["d"]), 0.0, case["side"])
    return mu, X, _inside(lo, hi, X).to(torch.uint8)


def _device_field(f):
    return pdmp.DeviceField(pdmp.RBF if f["kind"] == RBF else pdmp.RFF, f["centres"], f["w"], f["gamma"], f["phase"],
                            f["bias"])


L2 = 1e-4


def prepare(case, seed):
    op = case["op"]
    if op in ("morph", "grad", "logdet", "density", "query"):
        r, f, x, eta = _map(case, seed)
        st = {"op": op, "case": case, "field": _device_field(f), "x": x, "eta": eta}
        if op in ("morph", "logdet"):       # a program that calls again keeps its workspace
            st["ws"] = torch.empty(max(pdmp.morph_workspace(st["field"], case["N"]), 16), dtype=torch.uint8,
                                   device="cuda")
        if op == "morph":
            st["out"] = torch.empty_like(x)
        if op == "grad":
            st["g"] = r.normal(case["N"], case["d"])
            st["x"].requires_grad_(True)
            st["w"] = st["field"].w.clone().requires_grad_(True)
            st["bias"] = torch.tensor(f["bias"], device="cuda").requires_grad_(True)
        if op == "density":                 # points to be scored, inside the base box by more than the map moves them
            st["lo"], st["hi"] = [-0.5] * case["d"], [case["side"] + 0.5] * case["d"]
        return st
    if op == "batch":
        envs = [(_device_field(f), x, eta, case["T"]) for f, x, eta in _environments(case, seed)]
        b = pdmp.Batch(envs)
        b.prepare(0)
        return {"op": op, "batch": b}
    r = _Draws(seed)
    if op == "forward":
        net = pdmp.Surrogate([0.0] * 3, [5.0] * 3, [0.02] * 3, seed=int(seed))
        x = r.uniform((case["N"], 3), 0.0, 5.0)
        return {"op": op, "net": net, "x": x, "out": torch.empty_like(x)}
    if op == "train":                       # in the middle of a training run: the moments are warm
        net = pdmp.Surrogate([0.0] * 3, [5.0] * 3, [0.02] * 3, seed=int(seed))
        net.step = 500
        nw, nb = net.W.numel(), net.b.numel()
        m = 1e-3 * r.normal(nw + nb)
        v = 1e-5 * (0.5 + r.uniform((nw + nb,), 0.0, 1.0))
        net.adam.copy_(torch.cat([m[:nw], v[:nw], m[nw:], v[nw:]]))
        x, y = _pairs(r, case["B"])
        return {"op": op, "net": net, "x": x, "y": y, "loss": torch.zeros(1, device="cuda")}
    mu, X, y = _labelled(case, seed)
    fld = pdmp.DeviceField(pdmp.RBF, mu, torch.zeros(case["M"], device="cuda"), case["gamma"])
    return {"op": op, "case": case, "field": fld, "X": X, "y": y}


def run(s):
    op = s["op"]
    if op == "morph":
        return pdmp.morph(s["field"], s["x"], s["case"]["T"], s["eta"], out=s["out"], ws=s["ws"])
    if op == "grad":
        c = s["case"]
        y = pdmp.morph_autograd(s["field"], s["x"], c["T"], s["eta"], k=c["k"], w=s["w"], bias=s["bias"])
        gx, gw, gb = torch.autograd.grad(y, (s["x"], s["w"], s["bias"]), s["g"])
        return {"x_T": y.detach(), "x": gx, "w": gw, "bias": gb}
    if op == "logdet":
        ld, xT = pdmp.logdet(s["field"], s["x"], s["case"]["T"], s["eta"], want_xT=True, ws=s["ws"])
        return {"logdet": ld, "x_T": xT}
    if op == "density":
        lp, y = pdmp.log_density(s["field"], s["x"], s["case"]["T"], s["eta"], s["lo"], s["hi"])
        return {"log_p": lp, "y": y}
    if op == "batch":
        return list(s["batch"].run())
    if op == "forward":
        return s["net"].forward(s["x"], out=s["out"])
    if op == "train":
        loss = s["net"].train_step(s["x"], s["y"], lr=1e-4, loss=s["loss"])
        return {"loss": loss, "W": s["net"].W, "b": s["net"].b, "adam": s["net"].adam}
    if op == "fit":
        c = s["case"]
        w, bias, loss, alpha = pdmp.fit_occupancy(s["field"], s["X"], s["y"], L2, c["power"], c["iters"])
        return {"w": w, "bias": bias, "loss": loss, "alpha": alpha}
    return pdmp.occupancy_query(s["field"], s["x"])


# ------------------------------------------------------------------- what a pass cannot do without
def _evals(case):
    """Feature evaluations (one feature of one sample of one sweep) of a pass."""
    op = case["op"]
    if op == "batch":
        import random
        sizes, n = random.Random(1000 * case["envs"] + case["T"]), 0
        for _ in range(case["envs"]):
            sizes.choice((2, 3))
            n += sizes.randint(case["M_lo"], case["M_hi"]) * sizes.randint(case["N_lo"], case["N_hi"])
        return n * case["T"]
    if op == "fit":
        return case["n"] * case["M"] * 2 * (case["power"] + case["iters"])
    n = case["N"] * case["M"]
    return n if op == "query" else n * case["T"] * {"morph": 1, "logdet": 1, "density": 1, "grad": 3}[op]


def work(case):
    """Each input read once and each output written once; per feature evaluation the exponent (or the
    angle), the feature and its terms of s and grad s, with the Hessian's where a pass needs it."""
    op = case["op"]
    macs = 39 * 128 + 2 * 128 * 128 + 3 * 128
    if op == "forward":
        return {"bytes": 24 * case["N"] + 2 * macs, "flops": 2 * macs * case["N"]}
    if op == "train":
        p = macs + 3 * 128 + 3
        return {"bytes": 24 * case["B"] + 4 * 6 * p, "flops": 6 * macs * case["B"]}
    if op == "batch":
        import random
        sizes, b, fl = random.Random(1000 * case["envs"] + case["T"]), 0, 0
        for _ in range(case["envs"]):
            d = sizes.choice((2, 3))
            M, N = sizes.randint(case["M_lo"], case["M_hi"]), sizes.randint(case["N_lo"], case["N_hi"])
            b += 8 * N * d + 4 * M * (d + 1)
            fl += N * M * case["T"] * (4 * d + 4)
        return {"bytes": b, "flops": fl}
    d = case["d"]
    if op == "fit":
        return {"bytes": case["n"] * (4 * d + 1) + 4 * case["M"] * (d + 1), "flops": _evals(case) * (2 * d + 3)}
    per = 4 * d + 4 + (d * (d + 1) if op in ("logdet", "density") else 0)
    out = {"morph": 8 * d, "grad": 16 * d, "logdet": 8 * d + 4, "density": 8 * d + 4, "query": 8 * d + 8}[op]
    return {"bytes": case["N"] * out + 4 * case["M"] * (d + 2) * (2 if op == "grad" else 1), "flops": _evals(case) * per}


# ------------------------------------------------------------------- the same in 64 bits
MOST = {"morph": 6e10, "grad": 4e10, "logdet": 2e10, "density": 4e9, "batch": 6e10, "query": 4e10}


def _blocks(n, M):
    step = max(1, (1 << 25) // M)
    return [(i, min(n, i + step)) for i in range(0, n, step)]


def _grad_c(f, x):
    s, g, _ = _moments(f, x, hess=False)
    p = torch.sigmoid(s)
    return (p * (1.0 - p))[:, None] * g


def _exact_morph(f, x, T, eta):
    f, out = _double(f), torch.empty_like(x, dtype=torch.float64)
    for i, j in _blocks(x.shape[0], f["w"].shape[0]):
        y = x[i:j].double()
        for _ in range(T):
            y = y - eta * _grad_c(f, y)
        out[i:j] = y
    return out


def _log_det_step(f, x, eta):
    s, g, H = _moments(f, x)
    p = torch.sigmoid(s)
    d1 = p * (1.0 - p)
    J = -eta * (d1[:, None, None] * H + (d1 * (1.0 - 2.0 * p))[:, None, None] * (g[:, :, None] * g[:, None, :]))
    J = J + torch.eye(x.shape[1], dtype=x.dtype, device=x.device)
    return torch.linalg.slogdet(J)[1], x - eta * d1[:, None] * g


def _exact_grad(f, x, gT, T, eta):
    f = _double(f)
    w = f["w"].clone().requires_grad_(True)
    b = torch.tensor(f["bias"], dtype=torch.float64, device="cuda", requires_grad=True)
    f["w"], f["bias"] = w, b
    xT, g0 = torch.empty_like(x, dtype=torch.float64), torch.empty_like(x, dtype=torch.float64)
    gw, gb = torch.zeros_like(f["w"]), torch.zeros((), dtype=torch.float64, device="cuda")
    for i, j in _blocks(x.shape[0], 2 * w.shape[0]):
        xs = [x[i:j].double()]
        with torch.no_grad():
            for _ in range(T):
                xs.append(xs[-1] - eta * _grad_c(f, xs[-1]))
        a = gT[i:j].double()
        for y in reversed(xs[:-1]):
            y = y.requires_grad_(True)
            z = y - eta * _grad_c(f, y)
            a, dw, db = torch.autograd.grad(z, (y, w, b), a)
            gw += dw
            gb += db
        xT[i:j], g0[i:j] = xs[-1], a
    return {"x_T": xT, "x": g0, "w": gw, "bias": gb}


def _exact_density(f, z, T, eta, vol):
    f, lp, out = _double(f), torch.empty(z.shape[0], dtype=torch.float64, device="cuda"), torch.empty_like(z).double()
    for i, j in _blocks(z.shape[0], f["w"].shape[0]):
        x = z[i:j].double()
        acc = torch.zeros(j - i, dtype=torch.float64, device="cuda")
        for _ in range(T):
            t, y = x, x
            for _ in range(60):
                n = t + eta * _grad_c(f, y)
                done = bool((n - y).abs().max() < 1e-13)
                y = n
                if done:
                    break
            acc += _log_det_step(f, y, eta)[0]
            x = y
        out[i:j], lp[i:j] = x, -math.log(vol) - acc
    return {"log_p": lp, "y": out}


def _exact_fit(case, seed):
    mu, X, y = _labelled(case, seed)
    n, M = X.shape[0], mu.shape[0]
    P = torch.ones(n, M + 1, dtype=torch.float64, device="cuda")
    r2 = torch.zeros(n, M, dtype=torch.float64, device="cuda")
    for j in range(mu.shape[1]):
        r2 += (X[:, j:j + 1].double() - mu[:, j].double()) ** 2
    P[:, :M] = torch.exp(r2 * -case["gamma"])
    del r2
    lab = y.double()
    v = torch.full((M + 1,), 1.0 / math.sqrt(M + 1), dtype=torch.float64, device="cuda")
    lam = 0.0
    for _ in range(case["power"]):
        a = P.t() @ (P @ v) / n
        lam = float(a.norm())
        v = a / lam
    alpha = 1.0 / (0.25 * lam + L2)
    reg = torch.full((M + 1,), L2, dtype=torch.float64, device="cuda")
    reg[M] = 0.0
    w = torch.zeros(M + 1, dtype=torch.float64, device="cuda")
    prev = w
    for k in range(1, case["iters"] + 1):
        v = w + (k - 1) / (k + 2) * (w - prev)
        g = P.t() @ (torch.sigmoid(P @ v) - lab) / n + reg * v
        prev, w = w, v - alpha * g
    s = P @ w
    loss = (torch.nn.functional.softplus(s) - lab * s).mean() + 0.5 * L2 * (w[:M] ** 2).sum()
    return {"w": w[:M], "bias": float(w[M]), "loss": float(loss), "alpha": alpha}


def exact(case, seed):
    op = case["op"]
    if op in ("forward", "train"):          # BF16 networks: no 64-bit value
        return None
    if op == "fit":
        return _exact_fit(case, seed) if case["n"] * case["M"] < 1.2e9 else None
    if _evals(case) > MOST[op]:
        return None
    if op == "batch":
        return [_exact_morph(f, x, case["T"], eta) for f, x, eta in _environments(case, seed)]
    r, f, x, eta = _map(case, seed)
    if op == "morph":
        return _exact_morph(f, x, case["T"], eta)
    if op == "grad":
        return _exact_grad(f, x, r.normal(case["N"], case["d"]), case["T"], eta)
    f64 = _double(f)
    if op == "query":
        out = {"c": [], "s": [], "grad": []}
        for i, j in _blocks(case["N"], case["M"]):
            s, g, _ = _moments(f64, x[i:j].double(), hess=False)
            p = torch.sigmoid(s)
            out["c"].append(p)
            out["s"].append(s)
            out["grad"].append((p * (1.0 - p))[:, None] * g)
        return {k: torch.cat(v) for k, v in out.items()}
    if op == "logdet":
        ld, xT = torch.empty(case["N"], dtype=torch.float64, device="cuda"), torch.empty_like(x).double()
        for i, j in _blocks(case["N"], case["M"]):
            y, acc = x[i:j].double(), torch.zeros(j - i, dtype=torch.float64, device="cuda")
            for _ in range(case["T"]):
                l, y = _log_det_step(f64, y, eta)
                acc += l
            ld[i:j], xT[i:j] = acc, y
        return {"logdet": ld, "x_T": xT}
    return _exact_density(f, x, case["T"], eta, (case["side"] + 1.0) ** case["d"])
