"""The work that users of this library have it do, as cases to be timed and compared.

A case is a dict of plain numbers and texts. `listed()` gives twelve of them, `draw(rng)` one more
of the same ranges, `prepare(case, seed)` what a program has in hand before the call (plan,
potential, vectors), `run(state)` one pass through the public entry points, `work(case)` the
bytes and operations that the pass cannot do without, and `exact(case, seed)` what it returns,
in 64 bits by plain torch. The problems are those of `paper_2404_04507_gb300.workloads`.
"""
import math

import numpy as np
import torch

import paper_2404_04507_gb300 as iwf
from paper_2404_04507_gb300 import warmstart as ws
from paper_2404_04507_gb300 import workloads as W

DEV = "cuda:0"


def listed():
    return [
        # The smallest call: one apply of the 1D problem (24 x 32 grid) to its block of eight
        # vectors. Latency and launches are all of it.
        {"name": "apply_1d_f64", "kind": "apply", "problem": "qse1d", "K": 12, "L": 16,
         "eps": 1.0, "method": "iwfpm", "dtype": "f64", "nvec": 8},
        # The benchmark's step: 16 vectors on the 32^4 moire grid in complex double.
        {"name": "apply_moire32_f64", "kind": "apply", "problem": "moire", "K": 16, "L": 16,
         "eps": 0.5, "phases": False, "method": "iwfpm", "dtype": "f64", "nvec": 16},
        # The same block in complex float, with phases: the first phase of a mixed solve.
        {"name": "apply_moire32_c64", "kind": "apply", "problem": "moire", "K": 16, "L": 16,
         "eps": 5.0, "phases": True, "method": "iwfpm", "dtype": "c64", "nvec": 16},
        # A window of the sweep over cutoffs (22^4, no power of two) with its block of 24.
        {"name": "apply_sweep22_c64", "kind": "apply", "problem": "moire", "K": 11, "L": 11,
         "eps": 3.7, "phases": True, "method": "iwfpm", "dtype": "c64", "nvec": 24},
        # The 3D problem at its full size: 16^6 points, 16 vectors, complex float.
        {"name": "apply_3d16_c64", "kind": "apply", "problem": "qse3d", "K": 8, "L": 8,
         "eps": 3.0, "method": "iwfpm", "dtype": "c64", "nvec": 16},
        # Long axes: the projection-method reference of Example 4.1 (1280 x 2048).
        {"name": "apply_long_f64", "kind": "apply", "problem": "ex41", "K": 640, "L": 1024,
         "eps": 2.5, "method": "pm", "dtype": "f64", "nvec": 16},
        # A potential that is no sum of single-axis modes (81 modes on four axes at once) on a
        # ragged grid: the full potential grid and the transforms.
        {"name": "apply_modes_f64", "kind": "apply", "problem": "modes", "K": 9, "L": 11,
         "modes": 40, "radius": 2, "method": "iwfpm", "dtype": "f64", "nvec": 6},
        # The eigensolver's contractions on a long basis: G = S^H HS and X = S C.
        {"name": "contract_72x24", "kind": "contract", "nrows": 1 << 19, "m": 72, "q": 24},
        # The accuracy studies: a short solve for the ground state of Example 4.2 from a given
        # start block, its field on the observation grid, normalised, and its density.
        {"name": "ground_state_ex42", "kind": "ground", "K": 6, "L": 50, "block": 4,
         "maxit": 24, "rows": 1001},
        # The 16 lowest pairs at 32^4, six iterations from a given start block.
        {"name": "solve_moire32_f64", "kind": "solve", "K": 16, "L": 16, "eps": 0.5, "nev": 16,
         "block": 24, "maxit": 6},
        # A share of the sweep: problems with their own windows, strengths and phases in one
        # mixed-precision call, to convergence; eigenvalues are what the sweep keeps.
        {"name": "sweep_mixed", "kind": "sweep", "KLs": "5,6,7,6", "nev": 16, "block": 24},
        # One step of the warm-start network: loss and all gradients of a batch.
        {"name": "warmstart_step", "kind": "step", "hidden": 512, "layers": 4, "nvec": 16,
         "ncore": 256, "batch": 256},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _axis(half):
    """The next half-width from `half` whose axis the library takes: up to 32 points, or more
    with no prime factor above 7."""
    while True:
        n = 2 * half
        if n <= 32:
            return half
        for f in (2, 3, 5, 7):
            while n % f == 0:
                n //= f
        if n == 1:
            return half
        half += 1


def draw(rng):
    kind = rng.choice(["apply"] * 7 + ["contract", "ground", "solve", "sweep", "step"])
    if kind == "apply":
        problem = rng.choice(["qse1d", "moire", "moire", "qse3d", "ex41", "ex42", "modes"])
        c = {"kind": "apply", "problem": problem, "method": rng.choice(["iwfpm", "iwfpm", "pm"]),
             "dtype": rng.choice(["f64", "c64"])}
        if problem == "qse1d":
            c.update(K=rng.randint(4, 16), L=_axis(_log_int(rng, 8, 256)))
        elif problem == "moire":
            c.update(K=rng.randint(4, 16), L=rng.randint(4, 16), phases=rng.random() < 0.5)
        elif problem == "qse3d":
            c.update(K=rng.randint(2, 7), L=rng.randint(2, 7))
        elif problem == "ex41":
            c.update(K=_axis(_log_int(rng, 5, 640)), L=_axis(_log_int(rng, 20, 1024)))
        elif problem == "ex42":
            c.update(K=rng.randint(4, 10), L=_axis(_log_int(rng, 20, 512)))
        else:
            c.update(K=rng.randint(4, 13), L=rng.randint(4, 13), modes=rng.randint(24, 60),
                     radius=2)
        if problem != "modes":
            c["eps"] = round(rng.uniform(0.1, 10.0), 3)
        most = max(1, min(24, (1 << 26) // _points(c)))
        return dict(c, nvec=_log_int(rng, 1, most))
    if kind == "contract":
        return {"kind": "contract", "nrows": _log_int(rng, 1000, 1 << 19),
                "m": rng.randint(3, 72), "q": rng.randint(1, 24)}
    if kind == "ground":
        return {"kind": "ground", "K": rng.randint(4, 8), "L": _axis(rng.randint(16, 50)),
                "block": rng.choice([4, 8, 16]), "maxit": rng.randint(12, 24),
                "rows": rng.randint(33, 1001)}
    if kind == "solve":
        nev = rng.randint(4, 16)
        return {"kind": "solve", "K": rng.randint(5, 13), "L": rng.randint(5, 13),
                "eps": round(rng.uniform(0.3, 6.0), 3), "nev": nev,
                "block": min(24, nev + rng.randint(2, 8)), "maxit": rng.randint(5, 7)}
    if kind == "sweep":
        n = rng.randint(2, 3)
        return {"kind": "sweep", "KLs": ",".join(str(rng.choice([5, 5, 6])) for _ in range(n)),
                "nev": 16, "block": 24}
    return {"kind": "step", "hidden": 64 * rng.randint(2, 8), "layers": rng.randint(2, 4),
            "nvec": rng.choice([4, 8, 16]), "ncore": 32 * rng.randint(2, 8),
            "batch": 64 * rng.randint(1, 4)}


def _shape(c):
    d, n = {"qse1d": (1, 2), "moire": (2, 4), "qse3d": (3, 6), "ex41": (1, 2), "ex42": (2, 3),
            "modes": (2, 4)}[c["problem"]]
    return (2 * c["K"],) * d + (2 * c["L"],) * (n - d)


def _points(c):
    return math.prod(_shape(c))


def _problem(c, seed):
    """The problem of an apply case: phases and general modes come from the seed."""
    rng = np.random.default_rng(seed)
    K, L, kind, method = c["K"], c["L"], c["problem"], c["method"]
    if kind == "qse1d":
        return W.config_1d(K=K, L=L, eps=c["eps"], method=method)
    if kind == "moire":
        phases = rng.uniform(0.0, 2.0 * math.pi, size=4) if c["phases"] else None
        return W.config_moire(eps=c["eps"], K=K, L=L, method=method, phases=phases)
    if kind == "qse3d":
        pb = W.config_3d(eps=c["eps"], K=K, L=L)
        pb.method = method
        return pb
    if kind == "ex41":
        return W.example_41(c["eps"], K, L, method=method)
    if kind == "ex42":
        return W.example_42(0.8 * math.pi, 0.2 * math.pi, K, L, method=method)
    modes, coef = W.random_modes(4, c["modes"], c["radius"], seed=int(rng.integers(1 << 30)))
    return W.Problem("modes", W.moire_P(math.pi / 6), (K, K), (L, L), modes, coef, method=method)


def _plan(pb):
    p = iwf.Plan(pb.P, pb.K, pb.L, method=pb.method, shift_round=pb.shift_round)
    p.set_potential(pb.modes, pb.coef)
    return p


def _randn(shape, seed, dtype=torch.complex128):
    g = torch.Generator(device=DEV).manual_seed(seed)
    return torch.randn(shape, generator=g, dtype=dtype, device=DEV)


def _vectors(c, seed):
    x = _randn((c["nvec"], _points(c)), seed, torch.complex128 if c["dtype"] == "f64" else torch.complex64)
    return x.mul_(1.0 / math.sqrt(_points(c)))


def _sweep_problems(c, seed):
    rng = np.random.default_rng(seed)
    return [W.sweep_problem(rng.uniform(0.5, 10.0), rng.uniform(0.0, 2.0 * math.pi, size=4), int(k))
            for k in c["KLs"].split(",")]


def _dims(c):
    return [64] + [c["hidden"]] * c["layers"] + [2 * c["nvec"] * c["ncore"]]


def _network(c, seed):
    """Flat parameters, features and targets of one step: He-scaled weights, the features of
    potentials of the sweep, orthonormal target vectors."""
    rng = np.random.default_rng(seed)
    dims, flat = _dims(c), []
    for i, o in zip(dims[:-1], dims[1:]):
        flat += [rng.standard_normal(i * o, dtype=np.float32) * np.float32(math.sqrt(2.0 / i)),
                 rng.standard_normal(o, dtype=np.float32) * np.float32(0.05)]
    flat[-2] *= np.float32(0.1 / math.sqrt(c["ncore"]))
    flat[-1] *= np.float32(1.0 / math.sqrt(c["ncore"]))
    feat = W.warmstart_features(rng.uniform(0.1, 10.0, c["batch"]), rng.uniform(0.0, 2.0 * math.pi, (c["batch"], 4)))
    q, _ = torch.linalg.qr(_randn((c["batch"], c["ncore"], c["nvec"]), seed, torch.complex64))
    target = torch.view_as_real(q.transpose(1, 2).contiguous()).reshape(c["batch"], -1).contiguous()
    return np.concatenate(flat), torch.from_numpy(feat).to(DEV), target


def prepare(case, seed):
    c = case
    if c["kind"] == "apply":
        return {"kind": "apply", "plan": _plan(_problem(c, seed)), "x": _vectors(c, seed)}
    if c["kind"] == "contract":
        # an orthonormal-scale basis and its image: columns of different sizes, as H amplifies
        S = _randn((c["m"], c["nrows"]), seed).mul_(1.0 / math.sqrt(c["nrows"]))
        scale = torch.logspace(0, 2, c["m"], dtype=torch.float64, device=DEV)
        HS = _randn((c["m"], c["nrows"]), seed + 1).mul_(scale[:, None] / math.sqrt(c["nrows"]))
        return {"kind": "contract", "S": S, "HS": HS, "C": _randn((c["m"], c["q"]), seed + 2)}
    if c["kind"] == "ground":
        p = _plan(W.example_42(0.8 * math.pi, 0.2 * math.pi, c["K"], c["L"]))
        origin, step, count = W.grid_descriptor(2)
        # the middle rows of the observation grid; fields are compared at its centre
        skip = (count[0] - c["rows"]) // 2
        grid = ((origin[0] + skip * step[0], origin[1]), step, (c["rows"], count[1]))
        at = (count[0] // 2 - skip) * count[1] + count[1] // 2
        return {"kind": "ground", "plan": p, "X0": _start(p, c["block"], seed), "block": c["block"],
                "maxit": c["maxit"], "grid": grid, "at": at}
    if c["kind"] == "solve":
        pb = W.config_moire(eps=c["eps"], K=c["K"], L=c["L"])
        p = _plan(pb)
        return {"kind": "solve", "plan": p, "X0": _start(p, c["block"], seed), "nev": c["nev"],
                "block": c["block"], "maxit": c["maxit"], "probe": _randn((p.N,), seed + 1)}
    if c["kind"] == "sweep":
        return {"kind": "sweep", "plans": [_plan(pb) for pb in _sweep_problems(c, seed)],
                "nev": c["nev"], "block": c["block"], "seed": 1}
    flat, feat, target = _network(c, seed)
    net = ws.WarmStart(_dims(c), seed=1)
    net.set_params(flat)
    return {"kind": "step", "net": net, "feat": feat, "target": target, "nvec": c["nvec"], "ncore": c["ncore"]}


def _start(plan, block, seed):
    """A start block with the decay of low states: random, damped by the kinetic energy."""
    lam = torch.from_numpy(plan.kinetic()).to(DEV)
    return _randn((block, plan.N), seed).div_(1.0 + lam)


def run(state):
    s, kind = state, state["kind"]
    if kind == "apply":
        return s["plan"].apply(s["x"])
    if kind == "contract":
        return {"gram": iwf.gram(s["S"], s["HS"]), "update": iwf.block_update(s["S"], s["C"])}
    if kind == "ground":
        ev, X, _, _ = s["plan"].eigensolve(1, block=s["block"], maxit=s["maxit"], X0=s["X0"], raise_noconv=False)
        u = s["plan"].evaluate_grid(X[0], *s["grid"])
        rho, _ = s["plan"].normalize_field(u, at=s["at"])
        return {"E0": ev, "u": u, "rho": rho}
    if kind == "solve":
        ev, X, res, _ = s["plan"].eigensolve(s["nev"], block=s["block"], maxit=s["maxit"], X0=s["X0"], raise_noconv=False)
        # eigenvectors carry a free phase: fixed against a given vector
        z = X @ s["probe"].conj()
        return {"evals": ev, "resid": res, "evecs": X.mul_((z.conj() / z.abs())[:, None])}
    if kind == "sweep":
        ev, _, _, _, _ = iwf.batch_solve(s["plans"], s["nev"], block=s["block"], precision="c64", seed=s["seed"])
        return ev
    loss, grads = s["net"].loss_grad(s["feat"], s["target"], s["nvec"], s["ncore"])
    return {"loss": loss, "grads": grads}


def work(case):
    c = case
    if c["kind"] == "apply":
        # one read of psi and of Lambda, one write of H psi; per point the product with Lambda
        # and either the transforms' operations or one multiply-add per mode, the fewer of both
        N, elt = _points(c), 16 if c["dtype"] == "f64" else 8
        modes = 2 * c["modes"] if c["problem"] == "modes" else 2 * len(_shape(c))
        per = 4 + min(10 * math.log2(N) + 2, 8 * modes)
        return {"bytes": N * (2 * elt * c["nvec"] + elt / 2), "flops": N * c["nvec"] * per}
    if c["kind"] == "contract":
        n, m, q = c["nrows"], c["m"], c["q"]
        return {"bytes": 16.0 * n * (3 * m + q) + 16.0 * m * (m + 2 * q), "flops": 8.0 * n * m * (m + q)}
    if c["kind"] in ("ground", "solve"):
        moire = c["kind"] == "solve"
        N = (2 * c["K"]) ** 2 * (2 * c["L"]) ** (2 if moire else 1)
        b = c["block"]
        # an iteration reads X, P, W and their images and writes the next ones; its Gram and
        # update products of the 3b-column basis, and the products that keep it orthonormal
        by = c["maxit"] * N * b * 16.0 * 11
        fl = c["maxit"] * N * (8.0 * (9 * b * b / 2 + 4 * 3 * b * b + 2 * 2 * 2 * b * b + 2 * 3 * b * b) + 70.0 * b)
        if not moire:
            pts = c["rows"] * 1001
            by += 16.0 * 2 * pts + 8.0 * pts
            fl += 8.0 * 2 * c["L"] * pts * 2 * c["K"]
        return {"bytes": by, "flops": fl}
    if c["kind"] == "sweep":
        # about a hundred iterations of every problem
        N = sum((2 * int(k)) ** 4 for k in c["KLs"].split(","))
        b = c["block"]
        return {"bytes": 100.0 * N * b * 12 * 11, "flops": 100.0 * N * (8.0 * 30 * b * b + 70.0 * b)}
    d = _dims(c)
    weights = sum(i * o for i, o in zip(d[:-1], d[1:]))
    return {"bytes": 4.0 * (2 * weights + 2 * c["batch"] * d[-1]),
            "flops": 6.0 * c["batch"] * weights + 40.0 * c["batch"] * c["nvec"] ** 2 * c["ncore"]}


def _window(pb):
    """Slice bounds lo (slices x d), Lambda in window order, and for every window position its
    position in the periodic grid, by the window's definition."""
    d, n = pb.P.shape
    lens = [2 * k for k in pb.K] + [2 * l for l in pb.L]
    kII = np.stack(np.meshgrid(*[np.arange(-l, l) for l in pb.L], indexing="ij"), -1).reshape(-1, n - d)
    lo = np.tile(-np.asarray(pb.K, dtype=np.int64), (len(kII), 1))
    if pb.method != "pm":
        Q = np.linalg.inv(pb.P[:, :d]) @ pb.P[:, d:]
        shift = np.zeros((len(kII), d))
        for j in range(n - d):
            shift = shift + kII[:, j:j + 1] * Q[:, j]
        near = np.round(shift)
        shift = np.where(np.abs(shift - near) < 1e-9, near, shift)
        lo = np.ceil(-np.asarray(pb.K) - shift).astype(np.int64)
    lo, kII = torch.from_numpy(lo).to(DEV), torch.from_numpy(kII).to(DEV)
    o = [t.reshape(-1) for t in torch.meshgrid(*[torch.arange(v, device=DEV) for v in lens[:d]], indexing="ij")]
    star = torch.zeros((len(kII), len(o[0])), dtype=torch.int64, device=DEV)
    lam = torch.zeros((len(kII), len(o[0])), dtype=torch.float64, device=DEV)
    parts = [lo[:, j:j + 1] + o[j][None, :] for j in range(d)] + [kII[:, j:j + 1] for j in range(n - d)]
    for j in range(d, n):
        star = star * lens[j] + torch.remainder(parts[j], lens[j])
    for j in range(d):
        star = star * lens[j] + torch.remainder(parts[j], lens[j])
    for i in range(d):
        px = sum(float(pb.P[i, j]) * parts[j].double() for j in range(n))
        lam += 0.5 * px * px
    return lens[d:] + lens[:d], star.reshape(-1), lam.reshape(-1)


def exact(case, seed):
    c = case
    if c["kind"] == "apply":
        # H psi = Lambda psi + the cyclic convolution with the modes on the periodic grid
        pb, x = _problem(c, seed), _vectors(c, seed)
        d, n = pb.P.shape
        shape, star, lam = _window(pb)
        out = torch.empty(x.shape, dtype=torch.complex128, device=DEV)
        for v in range(x.shape[0]):
            psi = x[v].to(torch.complex128)
            grid = torch.empty_like(psi)
            grid[star] = psi
            grid = grid.reshape(shape)
            acc = torch.zeros_like(grid)
            for m, a in zip(pb.modes, pb.coef):
                m = [int(t) for t in m]
                acc += torch.roll(grid, m[d:] + m[:d], tuple(range(n))) * complex(a)
            out[v] = lam * psi + acc.reshape(-1)[star]
        return out
    if c["kind"] == "contract":
        s = prepare(c, seed)
        return {"gram": s["S"].conj() @ s["HS"].T, "update": s["C"].T @ s["S"]}
    if c["kind"] == "step":
        flat, feat, target = _network(c, seed)
        dims, at, layers = _dims(c), 0, []
        for i, o in zip(dims[:-1], dims[1:]):
            w = torch.from_numpy(flat[at:at + i * o].reshape(o, i)).to(DEV).double().requires_grad_()
            b = torch.from_numpy(flat[at + i * o:at + i * o + o]).to(DEV).double().requires_grad_()
            layers.append((w, b))
            at += i * o + o
        h = feat.double()
        for k, (w, b) in enumerate(layers):
            h = h @ w.T + b
            if k + 1 < len(layers):
                h = torch.nn.functional.gelu(h)
        size = (c["batch"], c["nvec"], c["ncore"])
        Y = torch.view_as_complex(h.reshape(*size, 2))
        X = torch.view_as_complex(target.double().reshape(*size, 2))
        xx, xy, yy = X.conj() @ X.transpose(1, 2), X.conj() @ Y.transpose(1, 2), Y.conj() @ Y.transpose(1, 2)
        loss = (xx.abs() ** 2 - 2 * xy.abs() ** 2 + yy.abs() ** 2).sum() / (c["batch"] * c["nvec"])
        loss.backward()
        grads = torch.cat([t.grad.reshape(-1) for wb in layers for t in wb])
        return {"loss": float(loss), "grads": grads}
    return None
