"""The work that users of this library have it do, as cases to be timed: solves
of Poisson systems in both precisions and both dimensions, batches of them, the
learned initial guess, and the gradients that train its network.

A case is a dict of plain values; its "kind" is one of
  solve   Solver.solve, run until the residual is below rtol (or, with "steps",
          for that many Arnoldi steps: the fixed budget of a real-time loop);
          "start" is "zero" (x0 = 0) or "prev" (x0 = the solution of the time
          step before, which is close to this step's);
  batch   Solver.solve_batch over systems of uneven sides;
  guess   Solver.guess: network, scaling and damped-Jacobi sweeps;
  train   Solver.nn_loss_grad: the loss of a minibatch and all gradients.
"""

import math

import numpy as np
import torch

from paper_2103_10975_gb300 import Solver

L2_BYTES = 126e6  # a basis beyond this streams from HBM in every pass


# ------------------------------------------------------------------ cases --
def listed():
    return [
        # the small validation problem: FP64, the library's default precision
        {"name": "solve_32_fp64", "kind": "solve", "dim": 2, "n": 32, "m": 20, "rtol": 1e-8,
         "precision": "fp64", "start": "zero", "steps": 0, "kappa": False, "tune": False},
        # plain FP64 GMRES(30) at the headline size: what the learned arm is judged against
        {"name": "solve_256_fp64", "kind": "solve", "dim": 2, "n": 256, "m": 30, "rtol": 1e-10,
         "precision": "fp64", "start": "zero", "steps": 0, "kappa": False, "tune": False},
        # one time step of the headline series: FP32 cycles, refined, from x_{t-1}
        {"name": "solve_256_fp32_prev", "kind": "solve", "dim": 2, "n": 256, "m": 30,
         "rtol": 1e-10, "precision": "fp32_refine", "start": "prev", "steps": 0, "kappa": False,
         "tune": False},
        # a small grid of odd side: rows off every alignment
        {"name": "solve_101_fp32", "kind": "solve", "dim": 2, "n": 101, "m": 30, "rtol": 1e-10,
         "precision": "fp32_refine", "start": "zero", "steps": 0, "kappa": False, "tune": False},
        # a middle size, basis too large for the SMs but not for L2; default options
        {"name": "solve_512_fp32_budget", "kind": "solve", "dim": 2, "n": 512, "m": 30,
         "rtol": 1e-10, "precision": "fp32_refine", "start": "prev", "steps": 300,
         "kappa": False, "tune": False},
        # the large refinement workload: the basis streams from HBM; tuned, as for production
        {"name": "solve_2048_fp32_budget", "kind": "solve", "dim": 2, "n": 2048, "m": 40,
         "rtol": 1e-10, "precision": "fp32_refine", "start": "prev", "steps": 200,
         "kappa": False, "tune": True},
        # the 3D variable-coefficient workload, tuned
        {"name": "cube_192_kappa_fp32_budget", "kind": "solve", "dim": 3, "n": 192, "m": 50,
         "rtol": 1e-10, "precision": "fp32_refine", "start": "prev", "steps": 100,
         "kappa": True, "tune": True},
        # a small 3D variable-coefficient system in FP64, odd side
        {"name": "cube_41_kappa_fp64", "kind": "solve", "dim": 3, "n": 41, "m": 30,
         "rtol": 1e-10, "precision": "fp64", "start": "zero", "steps": 0, "kappa": True,
         "tune": False},
        # independent instances of uneven sides in one launch
        {"name": "batch_40_fp32", "kind": "batch", "count": 40, "lo": 24, "hi": 160, "m": 30,
         "rtol": 1e-10, "precision": "fp32_refine"},
        # the learned guess of a time step at the headline size (32 sweeps, as in the benchmark)
        {"name": "guess_256", "kind": "guess", "dim": 2, "n": 256, "sweeps": 32},
        # the gradients of a training minibatch at the headline size and batch
        {"name": "train_256_b8", "kind": "train", "dim": 2, "n": 256, "batch": 8},
        # the same for the 3D network
        {"name": "train_cube_48_b2", "kind": "train", "dim": 3, "n": 48, "batch": 2},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["small", "small", "budget", "budget", "cube", "cube_budget", "batch",
                       "guess", "train", "train3"])
    prec = rng.choice(["fp64", "fp32_refine"])
    c = {"kind": "solve", "dim": 2, "rtol": 1e-10, "precision": prec, "steps": 0,
         "kappa": False, "tune": False}
    if kind == "small":
        # the basis fits the SMs: the range of sides, both precisions, both starts
        c.update(n=_log(rng, 24, 224 if prec == "fp64" else 288), m=rng.choice([20, 25, 30, 40]),
                 start=rng.choice(["zero", "prev"]))
    elif kind == "budget":
        # mid-size to large grids under a step budget
        n = _log(rng, 300, 1000 if prec == "fp64" else 2048)
        m = rng.choice([20, 30, 40])
        c.update(n=n, m=m, start="prev", steps=rng.choice([3, 4, 5]) * m, tune=n >= 1024)
    elif kind == "cube":
        # small 3D systems to convergence, with and without kappa
        c.update(dim=3, n=_log(rng, 14, 48), m=rng.choice([20, 30, 50]),
                 start=rng.choice(["zero", "prev"]), kappa=rng.random() < 0.7)
    elif kind == "cube_budget":
        # large 3D systems in FP32 under a step budget
        n = _log(rng, 64, 192)
        c.update(dim=3, n=n, m=rng.choice([30, 50]), precision="fp32_refine", start="prev",
                 steps=100, kappa=rng.random() < 0.7, tune=n >= 128)
    elif kind == "batch":
        lo = _log(rng, 16, 64)
        c = {"kind": "batch", "count": _log(rng, 6, 48), "lo": lo,
             "hi": min(176, lo + _log(rng, 16, 128)), "m": rng.choice([20, 30]), "rtol": 1e-10,
             "precision": "fp32_refine"}
    elif kind == "guess":
        c = {"kind": "guess", "dim": 2, "n": _log(rng, 40, 320), "sweeps": rng.choice([8, 16, 32])}
    elif kind == "train":
        c = {"kind": "train", "dim": 2, "n": _log(rng, 40, 256), "batch": rng.randint(1, 8)}
    else:
        c = {"kind": "train", "dim": 3, "n": _log(rng, 16, 56), "batch": rng.randint(1, 4)}
    return c


# ----------------------------------------------------------------- inputs --
def _coords(n):
    h = 2.0 / (n + 1)
    return -1.0 + h * torch.arange(1, n + 1, dtype=torch.float64, device="cuda")


def _bumps(n, dim, par):
    """Sum of Gaussians a exp(-|x - c|^2 / (2 s^2)), x the last axis; n^dim values."""
    x = _coords(n)
    out = torch.zeros((n,) * dim, dtype=torch.float64, device="cuda")
    for a, s, c in par:
        g = [torch.exp(-(x - ck) ** 2 / (2.0 * s * s)) for ck in c]
        t = torch.outer(g[1], g[0])
        out += a * (t if dim == 2 else g[2][:, None, None] * t)
    return out.reshape(-1)


def _sources(r, dim, count=3, s=0.1):
    """Charges of both signs; (now, a time step before): they move a little in between."""
    now, before = [], []
    for _ in range(count):
        c = r.uniform(-0.6, 0.6, dim)
        a = r.choice([-1.0, 1.0]) * r.uniform(0.5, 1.5)
        step = r.uniform(-1.0, 1.0, dim) * 0.005
        now.append((a, s, c))
        before.append((a * (1.0 + 0.005 * r.uniform(-1.0, 1.0)), s, c + step))
    return now, before


def _faces(n, dim, kappa):
    """Face coefficients along each axis (x first): n + 1 per line, walls included."""
    out = []
    for ax in range(dim):
        d = dim - 1 - ax
        lo, hi = kappa.narrow(d, 0, n - 1), kappa.narrow(d, 1, n - 1)
        out.append(torch.cat([kappa.narrow(d, 0, 1), 2.0 * lo * hi / (lo + hi),
                              kappa.narrow(d, n - 1, 1)], d))
    return out


def _apply(u, n, dim, faces=None):
    """A u on the n^dim grid with zero-Dirichlet walls, A = -div(kappa grad) / h^2, in FP64."""
    u = u.reshape((n,) * dim)
    out = torch.zeros_like(u)
    for ax in range(dim):
        d = dim - 1 - ax
        z = torch.zeros_like(u.narrow(d, 0, 1))
        p = torch.cat([z, u, z], d)
        flux = p.narrow(d, 1, n + 1) - p.narrow(d, 0, n + 1)
        if faces is not None:
            flux = faces[ax] * flux
        out -= flux.narrow(d, 1, n) - flux.narrow(d, 0, n)
    return (out * (0.25 * (n + 1) ** 2)).reshape(-1)


def _kappa(n, seed):
    """ln kappa: smooth Gaussian noise of unit deviation (correlation of 4 cells)."""
    g = torch.Generator(device="cuda").manual_seed(seed + 77)
    f = torch.randn((n,) * 3, dtype=torch.float64, device="cuda", generator=g)
    k = torch.exp(-torch.arange(-12, 13, dtype=torch.float64, device="cuda") ** 2 / 32.0)
    k = k / k.sum()
    i = torch.arange(n, device="cuda")
    band = (i[:, None] - i[None, :]).abs()
    S = k[(12 + band).clamp(max=24)] * (band <= 12)
    f = ((S @ f.reshape(n, -1)).reshape(n, n, n) @ S).transpose(1, 2) @ S
    return torch.exp(f / f.std()).float().contiguous()


def _poisson_2d(b, n):
    """A^-1 b for the 5-point Laplacian, by its sine eigenvectors."""
    i = torch.arange(1, n + 1, dtype=torch.float64, device="cuda")
    S = math.sqrt(2.0 / (n + 1)) * torch.sin(math.pi / (n + 1) * torch.outer(i, i))
    lam = (n + 1.0) ** 2 * torch.sin(math.pi * i / (2.0 * (n + 1))) ** 2
    return (S @ ((S @ b.reshape(n, n) @ S) / (lam[:, None] + lam[None, :])) @ S).reshape(-1)


def _system(case, seed):
    """(b, x0 or None, kappa or None) of a solve."""
    n, dim = case["n"], case["dim"]
    r = np.random.RandomState(seed % (1 << 31))
    kappa = _kappa(n, seed % (1 << 31)) if case["kappa"] else None
    now, before = _sources(r, dim)
    if case["start"] == "zero":
        return _bumps(n, dim, now), None, kappa
    if dim == 2 and not case["steps"]:
        return _bumps(n, dim, now), _poisson_2d(_bumps(n, dim, before), n), kappa
    # a smooth field that vanishes on the walls is the solution of the step
    # before; the sources then change by 1e-5 of their size (a fine time step)
    x = _coords(n)
    w = 1.0 - x * x
    wall = torch.outer(w, w) if dim == 2 else w[:, None, None] * torch.outer(w, w)
    x0 = wall.reshape(-1) * _bumps(n, dim, [(a, 0.3, c) for a, _, c in before])
    f = _faces(n, dim, kappa.double()) if kappa is not None else None
    b0 = _apply(x0, n, dim, f)
    d = _bumps(n, dim, now)
    b = b0 + 1e-5 * (b0.norm() / d.norm()) * d
    return b.contiguous(), x0.contiguous(), kappa


def _sides(case, seed):
    """The sides of a batch (the case's own: a program has its grids fixed) and the sources' stream."""
    g = np.random.RandomState(1000 * case["count"] + case["lo"] + case["hi"])
    ns = [int(v) for v in g.randint(case["lo"], case["hi"] + 1, case["count"])]
    return ns, np.random.RandomState(seed % (1 << 31))


def _levels(n):
    L = [n]
    while L[-1] // 2 >= 8:
        L.append(L[-1] // 2)
    return L


def _weights(n, dim, seed):
    """Weights as after some training, in the order in, level 0.., dilated, out: (w, b) each."""
    r = np.random.RandomState((seed + 5) % (1 << 31))
    k = (3,) * dim
    out = []
    for o, i in [(32, 1)] + [(32, 32)] * (len(_levels(n)) + 1) + [(1, 32)]:
        lim = math.sqrt(6.0 / (i * 3 ** dim))
        out.append((r.uniform(-lim, lim, (o, i) + k).astype(np.float32),
                    r.uniform(-0.1, 0.1, o).astype(np.float32)))
    return out


def _flat(ws):
    return np.concatenate([a.reshape(-1) for wb in ws for a in wb])


def _pairs(case, seed):
    """Normalised right-hand sides and unit-scale targets, as the replay ring holds them."""
    n, dim, B = case["n"], case["dim"], case["batch"]
    r = np.random.RandomState(seed % (1 << 31))
    u, t = [], []
    for _ in range(B):
        now, _ = _sources(r, dim)
        b = _bumps(n, dim, now)
        x = _poisson_2d(b, n) if dim == 2 else _bumps(n, dim, [(a, 0.4, c) for a, _, c in now])
        u.append(b / b.square().mean().sqrt())
        t.append(x / x.square().mean().sqrt())
    return torch.stack(u).float().contiguous(), torch.stack(t).float().contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "solve":
        b, x0, kappa = _system(case, seed)
        s = Solver(case["n"], dim=case["dim"], kappa=kappa, m=case["m"], rtol=case["rtol"],
                   precision=case["precision"], guess="zero" if x0 is None else "user",
                   max_iters=case["steps"] or 10 ** 7)
        if case["tune"]:
            s.autotune(b)
        return {"case": case, "solver": s, "b": b, "x0": x0, "x": torch.empty_like(b)}
    if kind == "batch":
        ns, r = _sides(case, seed)
        bs = [_bumps(n, 2, _sources(r, 2)[0]) for n in ns]
        s = Solver(case["hi"], m=case["m"], rtol=case["rtol"], precision=case["precision"],
                   batch_slots=4096)
        return {"case": case, "solver": s, "ns": ns, "bs": bs,
                "xs": [torch.empty_like(b) for b in bs]}
    n, dim = case["n"], case["dim"]
    if kind == "guess":
        s = Solver(n, dim=dim, m=30, precision="fp32_refine", guess="learned", batch=8,
                   guess_smooth=case["sweeps"])
        s.set_params(_flat(_weights(n, dim, seed)))
        b = _bumps(n, dim, _sources(np.random.RandomState(seed % (1 << 31)), dim)[0])
        return {"case": case, "solver": s, "b": b}
    s = Solver(n, dim=dim, m=30, precision="fp32_refine", guess="learned", batch=case["batch"])
    s.set_params(_flat(_weights(n, dim, seed)))
    u, t = _pairs(case, seed)
    return {"case": case, "solver": s, "u": u, "t": t}


def run(state):
    kind, s = state["case"]["kind"], state["solver"]
    if kind == "solve":
        if state["x0"] is not None:
            state["x"].copy_(state["x0"])
        return s.solve(state["b"], state["x"])[0]
    if kind == "batch":
        return s.solve_batch(state["ns"], state["bs"], state["xs"])[0]
    if kind == "guess":
        return s.guess(state["b"])
    loss, grad = s.nn_loss_grad(state["u"], state["t"])
    return {"loss": np.array([loss], dtype=np.float32), "grad": grad}


# ------------------------------------------------- what a pass has to do --
def _solve_work(n, dim, m, rtol, precision, start, steps):
    N = float(n) ** dim
    es = 8 if precision == "fp64" else 4
    if not steps:
        # restarted GMRES on the Laplacian: steps grow like n^2 / m (9900 at 256^2, m = 30)
        steps = 4.5 * n * n / m * (0.75 if start == "prev" else 1.0) * (math.log10(1 / rtol) / 10)
        steps = max(steps * (1.0 if dim == 2 else 0.7), 2.0 * n)
    # classical Gram-Schmidt twice: four multiply-adds per basis value and step
    flops = steps * N * (8.0 * (m / 2.0) + 12.0)
    nbytes = 8.0 * N * (2 if start == "zero" else 3)
    if (m + 1) * N * es > L2_BYTES:
        nbytes += steps * N * es * (m + 6.0)  # the basis, twice per step
    return nbytes, flops


def work(case):
    kind = case["kind"]
    if kind == "solve":
        b, f = _solve_work(case["n"], case["dim"], case["m"], case["rtol"], case["precision"],
                           case["start"], case["steps"])
        if case["kappa"]:
            b += 4.0 * case["n"] ** 3
    elif kind == "batch":
        side = 0.5 * (case["lo"] + case["hi"])
        b, f = _solve_work(side, 2, case["m"], case["rtol"], case["precision"], "zero", 0)
        b, f = b * case["count"], f * case["count"]
    else:
        n, dim = case["n"], case["dim"]
        B = case.get("batch", 1)
        taps = 3 ** dim
        pts = float(n) ** dim + sum(float(v) ** dim for v in _levels(n))  # dilated + levels
        f = 2.0 * taps * B * (1024.0 * pts + 64.0 * n ** dim)
        params = 4.0 * (1024 * taps + 32) * (len(_levels(n)) + 1) + 4.0 * (64 * taps + 33)
        if kind == "train":
            b = 8.0 * B * n ** dim + 2 * params
            f *= 3.0
        else:
            b = 16.0 * n ** dim + params
            f += 12.0 * case["sweeps"] * n ** dim
    return {"bytes": b, "flops": f}


# --------------------------------------------------------- in 64 bits ----
def _gmres(op, b, x, m, steps):
    """`steps` Arnoldi steps of GMRES(m) from x (classical Gram-Schmidt, twice)."""
    V = torch.empty((m + 1, b.numel()), dtype=torch.float64, device="cuda")
    while steps > 0:
        r = b - op(x)
        beta = r.norm()
        V[0] = r / beta
        k = min(m, steps)
        H = torch.zeros((k + 1, k), dtype=torch.float64, device="cuda")
        for j in range(k):
            w = op(V[j])
            for _ in range(2):
                h = V[: j + 1] @ w
                w = w - h @ V[: j + 1]
                H[: j + 1, j] += h
            H[j + 1, j] = w.norm()
            V[j + 1] = w / H[j + 1, j]
        e = np.zeros(k + 1)
        e[0] = float(beta)
        y = np.linalg.lstsq(H.cpu().numpy(), e, rcond=None)[0]
        x = x + torch.as_tensor(y, device="cuda") @ V[:k]
        steps -= k
    return x


def _cg(op, b):
    x = torch.zeros_like(b)
    r, p = b.clone(), b.clone()
    rr = r @ r
    stop = 1e-28 * float(rr)
    for it in range(5000):
        q = op(p)
        a = rr / (p @ q)
        x += a * p
        r -= a * q
        new = r @ r
        if it % 10 == 0 and float(new) < stop:
            break
        p = r + (new / rr) * p
        rr = new
    return x


def _network(n, dim, ws, u):
    """The network in FP64: u (B, n^dim) -> y (B, n^dim); ws: FP64 (w, b) tensors."""
    F = torch.nn.functional
    conv = F.conv2d if dim == 2 else F.conv3d
    pool = F.avg_pool2d if dim == 2 else F.avg_pool3d
    a = torch.relu(conv(u.reshape((-1, 1) + (n,) * dim), ws[0][0], ws[0][1], padding=1))
    s = 0.0
    L = _levels(n)
    for l in range(len(L)):
        z = torch.relu(conv(a, ws[1 + l][0], ws[1 + l][1], padding=1))
        s = s + (z if l == 0 else F.interpolate(z, size=(n,) * dim, align_corners=False,
                                                mode="bilinear" if dim == 2 else "trilinear"))
        if l + 1 < len(L):
            a = pool(a, 2)
    w, b = ws[len(L) + 1]
    t = s + torch.relu(conv(s, w, b, padding=2, dilation=2))
    w, b = ws[len(L) + 2]
    return conv(t, w, b, padding=1).reshape(u.shape)


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        n, dim = case["n"], case["dim"]
        b, x0, kappa = _system(case, seed)
        f = _faces(n, dim, kappa.double()) if kappa is not None else None
        if case["steps"]:
            return _gmres(lambda u: _apply(u, n, dim, f), b, x0, case["m"], case["steps"])
        if dim == 2:
            return _poisson_2d(b, n)
        return _cg(lambda u: _apply(u, n, dim, f), b)
    if kind == "batch":
        ns, r = _sides(case, seed)
        return [_poisson_2d(_bumps(n, 2, _sources(r, 2)[0]), n) for n in ns]
    n, dim = case["n"], case["dim"]
    ws = [(torch.as_tensor(w, device="cuda").double().requires_grad_(),
           torch.as_tensor(b, device="cuda").double().requires_grad_())
          for w, b in _weights(n, dim, seed)]
    if kind == "train":
        u, t = _pairs(case, seed)
        loss = (_network(n, dim, ws, u.double()) - t.double()).square().mean()
        g = torch.autograd.grad(loss, [p for wb in ws for p in wb])
        return {"loss": loss.detach().reshape(1),
                "grad": torch.cat([p.reshape(-1) for p in g])}
    b = _bumps(n, dim, _sources(np.random.RandomState(seed % (1 << 31)), dim)[0])
    s = b.square().mean().sqrt()
    with torch.no_grad():
        x = s * _network(n, dim, ws, (b / s)[None])[0]
        f = np.float64(np.float32(0.8)) / (n + 1.0) ** 2  # omega over the diagonal of A
        for _ in range(case["sweeps"]):
            x = x + f * (b - _apply(x, n, dim))
    return x
