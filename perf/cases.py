"""The workloads whose speed and accuracy are measured, each one pass through
the package's public entry points on particles of the models it is used with.

``listed()`` gives the fixed cases, ``draw(rng)`` more of the same ranges,
``prepare`` what a program holds before the call, ``run`` the call,
``work`` the bytes and operations it cannot do without and ``exact`` the same
outputs in 64-bit torch arithmetic from the formulas alone.

The coefficients of a mixed-precision force calculation are an intermediate
(FP32 basis values summed into doubles), so those cases return the force;
the FP64 cases return the coefficients as well.
"""
from __future__ import annotations

import math
import random

import torch

from paper_1406_4254_gb300 import autotune, etics

DT = 0.01           # leapfrog step of the Plummer run
DT_BAR = 0.005      # leapfrog step of the bar-perturbed run


def listed():
    return [
        # one small system (a cluster, a test particle set): launches and latency count
        {"name": "scf_small", "kind": "scf", "dtype": "f32", "basis": "ho", "N": 4219,
         "n_max": 10, "l_max": 6},
        # the plain double-precision SCF force of a small Hernquist sphere
        {"name": "scf_fp64", "kind": "scf", "dtype": "f64", "basis": "ho", "N": 16384,
         "n_max": 10, "l_max": 6},
        # an expansion order and a size that no kernel is written for
        {"name": "scf_general", "kind": "scf", "dtype": "f32", "basis": "ho", "N": 200003,
         "n_max": 8, "l_max": 4},
        # the alternative radial basis on the model it is made for
        {"name": "scf_clutton_brock", "kind": "scf", "dtype": "f32", "basis": "cb", "N": 262144,
         "n_max": 10, "l_max": 6},
        # time integration of a Plummer sphere: one kick-drift-kick step
        {"name": "leapfrog_plummer", "kind": "leapfrog", "dtype": "f32", "model": "plummer",
         "N": 1 << 20, "n_max": 10, "l_max": 6},
        # the bar-perturbed Hernquist sphere at a high order: one plain step of a large run
        {"name": "leapfrog_bar", "kind": "leapfrog", "dtype": "f32", "model": "bar",
         "N": 1 << 24, "n_max": 14, "l_max": 8},
        # MEX of one small system: a chain of dependent launches
        {"name": "mex_small", "kind": "mex", "dtype": "f32", "N": 10007, "l_max": 4},
        # the MEX force of the flattened Hernquist model at the benchmark's size
        {"name": "mex_flattened", "kind": "mex", "dtype": "f32", "N": 1 << 20, "l_max": 6},
        # MEX at the highest order of the accuracy study, a ragged size
        {"name": "mex_l10", "kind": "mex", "dtype": "f32", "N": 500009, "l_max": 10},
        # the double-precision MEX force
        {"name": "mex_fp64", "kind": "mex", "dtype": "f64", "N": 100003, "l_max": 6},
        # an ensemble of independent systems of uneven size and order in one call
        {"name": "batch_ensemble", "kind": "batch", "dtype": "f32", "systems": 256, "ensemble": 0},
        # one training iteration of the coefficient-forecasting network: 16
        # histories of 1215 coefficients, loss, gradients and the Adam update
        {"name": "mlp_training", "kind": "mlp", "rows": 16 * 1215, "hidden": 256, "outputs": 3},
    ]


def _size(rng: random.Random, lo: float, hi: float) -> int:
    """A size between 2^lo and 2^hi, uniform in its logarithm; three of four odd."""
    n = int(round(2.0 ** rng.uniform(lo, hi)))
    return n if rng.random() < 0.25 else n | 1


def draw(rng: random.Random):
    kind = rng.choice(["scf", "scf", "scf_cb", "scf64", "leapfrog", "mex", "mex", "mex64", "batch",
                       "mlp"])
    if kind == "scf":
        return {"kind": "scf", "dtype": "f32", "basis": "ho", "N": _size(rng, 12, 21),
                "n_max": rng.randint(4, 16), "l_max": rng.randint(0, 10)}
    if kind == "scf_cb":
        return {"kind": "scf", "dtype": "f32", "basis": "cb", "N": _size(rng, 12, 20),
                "n_max": rng.randint(4, 14), "l_max": rng.randint(0, 8)}
    if kind == "scf64":
        return {"kind": "scf", "dtype": "f64", "basis": "ho", "N": _size(rng, 12, 16),
                "n_max": rng.randint(4, 14), "l_max": rng.randint(0, 8)}
    if kind == "leapfrog":
        n_max, l_max = rng.choice([(10, 6), (14, 8), (rng.randint(4, 14), rng.randint(0, 8))])
        return {"kind": "leapfrog", "dtype": "f32", "model": rng.choice(["plummer", "bar"]),
                "N": _size(rng, 14, 22), "n_max": n_max, "l_max": l_max}
    if kind == "mex":
        return {"kind": "mex", "dtype": "f32", "N": _size(rng, 12, 22), "l_max": rng.randint(0, 10)}
    if kind == "mex64":
        return {"kind": "mex", "dtype": "f64", "N": _size(rng, 12, 17), "l_max": rng.randint(0, 6)}
    if kind == "batch":
        return {"kind": "batch", "dtype": "f32", "systems": rng.randint(16, 128),
                "ensemble": rng.randint(1, 1 << 20)}
    return {"kind": "mlp", "rows": 1215 * rng.randint(4, 32), "hidden": rng.choice([64, 128, 256]),
            "outputs": rng.randint(1, 4)}


# ---- inputs -------------------------------------------------------------------
def _gen(seed: int) -> torch.Generator:
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _isotropic(g, n):
    ct = 2.0 * _rand(g, n) - 1.0
    ph = 2.0 * math.pi * _rand(g, n)
    st = torch.sqrt((1.0 - ct * ct).clamp_min(0.0))
    return torch.stack([st * torch.cos(ph), st * torch.sin(ph), ct], dim=1)


def _posm(x, n):
    return torch.cat([x, torch.full((x.shape[0], 1), 1.0 / n, dtype=torch.float64, device="cuda")],
                     dim=1)


def _hernquist(g, n, axes=(1.0, 1.0, 1.0), bar=0.0):
    su = torch.sqrt(_rand(g, n))
    r = su / (1.0 - su)
    d = _isotropic(g, n)
    if bar:
        # density 1 + bar sin^2(theta) cos(2 phi): directions redrawn once
        # where a rejection test fails (the small bias left is of second order)
        w = 1.0 + bar * (d[:, 0] ** 2 - d[:, 1] ** 2)
        d = torch.where((_rand(g, n) * (1.0 + bar) < w)[:, None], d, _isotropic(g, n))
    return _posm(d * r[:, None] * torch.tensor(axes, dtype=torch.float64, device="cuda"), n)


def _plummer(g, n):
    u = _rand(g, n).clamp_min(1e-12)
    r = 1.0 / torch.sqrt(u ** (-2.0 / 3.0) - 1.0)
    return _posm(_isotropic(g, n) * r[:, None], n)


def _velocities(g, posm, escape2):
    """Isotropic velocities below the escape speed (squared: escape2), speed
    fraction q with density q^2 (1 - q^2)^(7/2): q^2 is Beta(3/2, 9/2)."""
    n = posm.shape[0]
    cand = _rand(g, n, 12)                      # rejection: the first accepted of 12
    ok = _rand(g, n, 12) * 0.1 < cand ** 2 * (1.0 - cand ** 2) ** 3.5
    q = torch.gather(cand, 1, ok.to(torch.int8).argmax(dim=1, keepdim=True))[:, 0]
    v = torch.zeros_like(posm)
    v[:, :3] = _isotropic(g, n) * (q * torch.sqrt(escape2))[:, None]
    return v


def _ensemble(case):
    """Sizes and orders of the systems: N log-uniform in [2^12, 2^18], n_max
    in 6..14, l_max in 2..8."""
    rng = random.Random(case["ensemble"])
    k = case["systems"]
    return ([int(round(2.0 ** rng.uniform(12, 18))) for _ in range(k)],
            [rng.randint(6, 14) for _ in range(k)], [rng.randint(2, 8) for _ in range(k)])


def _dtype(case):
    return torch.float32 if case["dtype"] == "f32" else torch.float64


def _particles(case, seed):
    """The case's particles (and velocities) in its own precision, from the seed alone."""
    g = _gen(seed)
    kind = case["kind"]
    if kind == "scf":
        p = _plummer(g, case["N"]) if case["basis"] == "cb" else _hernquist(g, case["N"],
                                                                            (1.0, 0.8, 0.6))
        return p.to(_dtype(case)), None
    if kind == "mex":
        return _hernquist(g, case["N"], (1.0, 0.8, 0.6)).to(_dtype(case)), None
    if kind == "leapfrog":
        if case["model"] == "plummer":
            p = _plummer(g, case["N"])
            esc = 2.0 / torch.sqrt(1.0 + (p[:, :3] ** 2).sum(dim=1))
        else:
            p = _hernquist(g, case["N"], bar=0.05)
            esc = 2.0 / (1.0 + (p[:, :3] ** 2).sum(dim=1).sqrt())
        v = _velocities(g, p, esc)
        return p.to(_dtype(case)), v.to(_dtype(case))
    sizes = _ensemble(case)[0]
    p = _hernquist(g, sum(sizes))
    p[:, 3] = torch.cat([torch.full((n,), 1.0 / n, dtype=torch.float64, device="cuda")
                         for n in sizes])
    return p.to(_dtype(case)), None


def _mlp_inputs(case, seed):
    """A network in the middle of its training: parameters, moments, a minibatch."""
    g = _gen(seed)
    dims = [8, case["hidden"], case["hidden"], case["outputs"]]

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float32)

    parts = []
    for i in range(3):
        parts += [normal(dims[i] * dims[i + 1]) / math.sqrt(dims[i]), 0.1 * normal(dims[i + 1])]
    params = torch.cat(parts)
    m = 1e-3 * normal(params.numel())
    v = (1e-3 * (0.5 + torch.rand(params.numel(), generator=g, device="cuda"))) ** 2
    x = normal(case["rows"], 8).to(torch.bfloat16)
    # what the predictors miss: mostly noise, a part that the features carry
    t = normal(case["rows"], case["outputs"]) + 0.3 * x.float().sum(dim=1, keepdim=True)
    return dims, params, m, v, x, t


def _dt(case):
    return DT if case["model"] == "plummer" else DT_BAR


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "mlp":
        dims, params, m, v, x, t = _mlp_inputs(case, seed)
        s.update(dims=dims, params=params, m=m, v=v, x=x, target=t, t=500,
                 params_bf16=torch.empty(params.numel(), dtype=torch.bfloat16, device="cuda"),
                 grads=torch.empty_like(params),
                 loss=torch.empty(1, dtype=torch.float64, device="cuda"),
                 ws=etics.mlp_workspace(dims, case["rows"]))
        etics.mlp_to_bf16(dims, params, s["params_bf16"])
        return s
    s["posm"], vel = _particles(case, seed)
    if kind == "leapfrog":
        s["vel"] = vel
        s["acc"], _ = etics.scf_force(s["posm"], case["n_max"], case["l_max"])
    if kind == "batch":
        sizes, nm, lm = _ensemble(case)
        s["plan"] = etics.BatchPlan(sizes, nm, lm, tuning=autotune.lookup(nm, lm, sizes))
    return s


# ---- the measured calls ---------------------------------------------------------
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "scf":
        basis = etics.BASIS_CB if case["basis"] == "cb" else etics.BASIS_HO
        out, c = etics.scf_force(state["posm"], case["n_max"], case["l_max"], basis=basis)
        return {"accpot": out, "coeffs": c} if case["dtype"] == "f64" else {"accpot": out}
    if kind == "mex":
        return {"accpot": etics.mex_field(state["posm"], case["l_max"])}
    if kind == "leapfrog":
        etics.leapfrog_step(state["posm"], state["vel"], state["acc"], _dt(case), etics.SCF,
                            case["n_max"], case["l_max"])
        return {"posm": state["posm"], "vel": state["vel"], "accpot": state["acc"]}
    if kind == "batch":
        _, out = etics.scf_batch(state["posm"], state["plan"])
        return {"accpot": out}
    state["t"] += 1
    etics.mlp_loss_grad(state["dims"], state["params"], state["params_bf16"], state["x"],
                        state["target"], state["grads"], state["loss"], ws=state["ws"])
    etics.mlp_adam(state["dims"], state["params"], state["grads"], state["m"], state["v"],
                   state["t"], 1e-3, state["params_bf16"])
    return {k: state[k] for k in ("loss", "grads", "params", "m", "v")}


# ---- what a pass cannot do without ------------------------------------------------
def _scf_flops(n, n_max, l_max):
    cols = (l_max + 1) ** 2
    rad = (n_max + 1) * (l_max + 1)
    coeff = 2 * (n_max + 1) * cols + 3 * rad + 4 * cols + 30
    field = 4 * (n_max + 1) * cols + 6 * rad + 10 * cols + 8 * (l_max + 1) + 80
    return n * (coeff + field)


def work(case):
    kind = case["kind"]
    if kind == "mlp":
        h, o, b = case["hidden"], case["outputs"], case["rows"]
        params = 8 * h + h + h * h + h + h * o + o
        products = 8 * h + h * h + h * o
        # forward, weight gradients, and the error of the two upper layers
        flops = 2 * b * (2 * products + h * h + h * o)
        return {"bytes": b * (16 + 4 * o) + params * (4 * 4 + 4 * 4 + 2), "flops": flops}
    size = 16 if case["dtype"] == "f32" else 32
    if kind == "batch":
        sizes, nm, lm = _ensemble(case)
        return {"bytes": 2 * size * sum(sizes),
                "flops": sum(_scf_flops(n, a, b) for n, a, b in zip(sizes, nm, lm))}
    n, l_max = case["N"], case["l_max"]
    if kind == "mex":
        return {"bytes": 2 * size * n, "flops": n * (42 * (l_max + 1) ** 2 + 40)}
    vectors = 6 if kind == "leapfrog" else 2
    return {"bytes": vectors * size * n, "flops": _scf_flops(n, case["n_max"], l_max)}


# ---- the same outputs in 64 bits ---------------------------------------------------
def _solid(x, l_max):
    """Real orthonormal solid harmonics r^l Y_lm of the points x (N, 3), a
    list over l of (2l+1, N) stacks in the order m = -l..l."""
    cx, cy, cz = x[:, 0], x[:, 1], x[:, 2]
    r2 = cx * cx + cy * cy + cz * cz
    one = torch.ones_like(cx)
    c = {(0, 0): one}
    s = {(0, 0): torch.zeros_like(cx)}
    out = []
    for l in range(l_max + 1):
        if l:
            d = 2.0 * l - 1.0
            c[l, l] = d * (cx * c[l - 1, l - 1] - cy * s[l - 1, l - 1])
            s[l, l] = d * (cx * s[l - 1, l - 1] + cy * c[l - 1, l - 1])
            for m in range(l):
                for t in (c, s):
                    up = d * cz * t[l - 1, m]
                    t[l, m] = (up - (l + m - 1.0) * r2 * t[l - 2, m] if l - 2 >= m else up) / (l - m)
        k = [math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - m) / math.factorial(l + m) *
                       (2.0 if m else 1.0)) for m in range(l + 1)]
        out.append(torch.stack([k[m] * s[l, m] for m in range(l, 0, -1)] +
                               [k[m] * c[l, m] for m in range(l + 1)]))
    return out


def _radial(r, n_max, l, basis):
    """phi_nl(r) / r^l for n = 0..n_max: (n_max + 1, N)."""
    if basis == "cb":
        xi, pre, alpha = (r * r - 1) / (r * r + 1), -(1 + r * r) ** (-(l + 0.5)), l + 1.0
    else:
        xi, pre, alpha = (r - 1) / (r + 1), -(1 + r) ** (-(2.0 * l + 1)), 2 * l + 1.5
    c = [torch.ones_like(r)]
    if n_max:
        c.append(2 * alpha * xi)
    for n in range(2, n_max + 1):
        c.append((2 * (n + alpha - 1) * xi * c[n - 1] - (n + 2 * alpha - 2) * c[n - 2]) / n)
    return torch.stack([pre * v for v in c])


def _norm(n, l, basis):
    lg = math.lgamma
    if basis == "cb":
        k = 4.0 * n * (n + 2 * l + 2) + (2 * l + 1) * (2 * l + 3)
        return -k * math.exp(lg(n + 2 * l + 2) - lg(n + 1) - 2 * lg(l + 1) -
                             (4 * l + 6) * math.log(2)) / (n + l + 1)
    k = n * (n + 4 * l + 3) / 2.0 + (l + 1) * (2 * l + 1)
    return -k * math.exp(lg(n + 4 * l + 3) - lg(n + 1) - 2 * lg(2 * l + 1.5) -
                         (8 * l + 6) * math.log(2)) / (n + 2 * l + 1.5)


_CHUNK = 1 << 18


def _scf_exact(p, n_max, l_max, basis):
    """(accpot, coefficients) of the particles p (N, 4) in 64 bits."""
    inv = [torch.tensor([1.0 / _norm(n, l, basis) for n in range(n_max + 1)], dtype=torch.float64,
                        device=p.device) for l in range(l_max + 1)]
    coef = [0.0] * (l_max + 1)
    for q in p.split(_CHUNK):
        r = q[:, :3].norm(dim=1)
        z = _solid(q[:, :3], l_max)
        for l in range(l_max + 1):
            coef[l] = coef[l] + (_radial(r, n_max, l, basis) * q[:, 3]) @ z[l].T
    coef = [inv[l][:, None] * coef[l] for l in range(l_max + 1)]
    out = torch.empty_like(p)
    for q, o in zip(p.split(_CHUNK), out.split(_CHUNK)):
        x = q[:, :3].clone().requires_grad_(True)
        with torch.enable_grad():
            r = x.norm(dim=1)
            z = _solid(x, l_max)
            pot = 0.0
            for l in range(l_max + 1):
                pot = pot + ((coef[l].T @ _radial(r, n_max, l, basis)) * z[l]).sum(dim=0)
            grad, = torch.autograd.grad(pot.sum(), x)
        o[:, :3] = -grad
        o[:, 3] = pot.detach()
    return out, torch.cat(coef, dim=1)


def _mex_exact(p, l_max):
    r2 = (p[:, 0] * p[:, 0] + p[:, 1] * p[:, 1]) + p[:, 2] * p[:, 2]
    order = torch.sort(r2, stable=True).indices
    q = p[order]
    r = q[:, :3].norm(dim=1)
    inner, outer = [], []
    for l, z in enumerate(_solid(q[:, :3], l_max)):
        m_in = z * q[:, 3]
        m_out = m_in * r ** (-(2.0 * l + 1))
        inner.append(torch.nn.functional.pad(m_in.cumsum(dim=1)[:, :-1], (1, 0)))
        outer.append(torch.nn.functional.pad(m_out.flip(1).cumsum(dim=1).flip(1)[:, 1:], (0, 1)))
    srt = torch.empty_like(q)
    for i in range(0, q.shape[0], _CHUNK):
        e = min(i + _CHUNK, q.shape[0])
        x = q[i:e, :3].clone().requires_grad_(True)
        with torch.enable_grad():
            rr = x.norm(dim=1)
            pot = 0.0
            for l, z in enumerate(_solid(x, l_max)):
                k = -4.0 * math.pi / (2 * l + 1)
                pot = pot + k * ((inner[l][:, i:e] * rr ** (-(2.0 * l + 1)) + outer[l][:, i:e]) *
                                 z).sum(dim=0)
            grad, = torch.autograd.grad(pot.sum(), x)
        srt[i:e, :3] = -grad
        srt[i:e, 3] = pot.detach()
    out = torch.empty_like(srt)
    out[order] = srt
    return out


def _mlp_exact(case, seed):
    dims, params, m, v, x, target = _mlp_inputs(case, seed)
    p = params.double().requires_grad_(True)
    with torch.enable_grad():
        h, o = x.double(), 0
        for i in range(3):
            a, b = dims[i], dims[i + 1]
            h = h @ p[o:o + a * b].view(a, b) + p[o + a * b:o + a * b + b]
            o += a * b + b
            if i < 2:
                h = torch.tanh(h)
        loss = ((h - target.double()) ** 2).mean()
        g, = torch.autograd.grad(loss, p)
    t, lr, b1, b2, eps = 501, 1e-3, 0.9, 0.999, 1e-8
    m = b1 * m.double() + (1 - b1) * g
    v = b2 * v.double() + (1 - b2) * g * g
    new = p.detach() - lr * (m / (1 - b1 ** t)) / (torch.sqrt(v / (1 - b2 ** t)) + eps)
    return {"loss": loss.detach().reshape(1), "grads": g, "params": new, "m": m, "v": v}


def exact(case, seed):
    kind = case["kind"]
    if kind == "mlp":
        return _mlp_exact(case, seed)
    posm, vel = _particles(case, seed)
    p = posm.double()
    if kind == "scf":
        acc, c = _scf_exact(p, case["n_max"], case["l_max"], case["basis"])
        return {"accpot": acc, "coeffs": c} if case["dtype"] == "f64" else {"accpot": acc}
    if kind == "mex":
        return {"accpot": _mex_exact(p, case["l_max"])}
    if kind == "leapfrog":
        dt, v = _dt(case), vel.double()
        acc, _ = _scf_exact(p, case["n_max"], case["l_max"], "ho")
        v[:, :3] += 0.5 * dt * acc[:, :3]
        p[:, :3] += dt * v[:, :3]
        acc, _ = _scf_exact(p, case["n_max"], case["l_max"], "ho")
        v[:, :3] += 0.5 * dt * acc[:, :3]
        return {"posm": p, "vel": v, "accpot": acc}
    parts, o = [], 0
    for n, a, b in zip(*_ensemble(case)):
        parts.append(_scf_exact(p[o:o + n], a, b, "ho")[0])
        o += n
    return {"accpot": torch.cat(parts)}
