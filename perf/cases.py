"""The work a program has this library do, as cases that can be timed and compared.

Every case is one call, or one short sequence of calls, of the public binding on device tensors:
a single evaluation in each precision from a few hundred to 100 000 charges, a batch of many
systems, separate evaluation points, and the energy with its derivatives.  Sizes, boxes and
(p, M) settings are those of the package's workloads, of the tests and of the benchmark, with
odd sizes among them.

`exact` restates the method in plain torch and numpy float64 (direct image sums, least squares by
SVD, closed-form box mean) for the sizes where that takes seconds.
"""
from __future__ import annotations

import math
import types

import numpy as np
import torch

from paper_1310_4374_gb300 import binding as B
from paper_1310_4374_gb300 import workloads as W
from paper_1310_4374_gb300.autograd import PeriodicCoulombEnergy

DEV = "cuda:0"
PM = {8: 200, 12: 400, 16: 800}               # degree -> check points, the batch workload's settings
BOXES = ((1.0, 1.0, 1.0), (1.0, 1.5, 2.0), (1.0, 1.0, 2.0))


def _single(name, api, precision, N, d, p, charges="gauss", **more):
    c = {"name": name, "api": api, "precision": precision, "N": N, "d1": d[0], "d2": d[1], "d3": d[2], "p": p,
         "M": PM[p], "charges": charges}
    c.update(more)
    return c


def listed():
    cube, box, long = BOXES
    return [
        # the smallest system of the batch workload on its own, replayed step after step by a
        # simulation loop (fixed buffers, CUDA graph): latency and launches are everything
        _single("fp32c_500_graph", "graph", "fp32c", 500, cube, 8, "pm1"),
        # random +-1 charges in the unit cube in the default precision, called the documented way
        _single("fp64_1000_call", "call", "fp64", 1000, cube, 8, "pm1"),
        # the rock-salt lattice with thermal jitter (16^3 ions), float64
        _single("fp64_lattice_4096", "eval", "fp64", 4096, cube, 12, "lattice"),
        # an ordinary molecular system, an odd size just under the symmetric kernel's threshold
        _single("fp32c_5001", "eval", "fp32c", 5001, box, 12),
        # the largest system of the batch workload on its own, ragged
        _single("fp32c_19999", "eval", "fp32c", 19999, box, 16),
        # the precision workload: 1e5 charges in a rectangular box, the benchmark's default step
        _single("fp32c_100000", "eval", "fp32c", 100000, box, 16),
        # float64 at a size where the pair sum is all
        _single("fp64_12001", "eval", "fp64", 12001, box, 12),
        # float64-class results on the float32 pipe (the precision workload's second arm)
        _single("ff_20011", "eval", "ff", 20011, box, 16),
        # many systems of uneven size, box and degree in one graph replay
        {"name": "batch_32", "api": "batch", "precision": "fp32c", "systems": 32, "n_lo": 500, "n_hi": 20000,
         "shape": 3},
        # potential and field of the charges at other points of the box (a probe grid, a new configuration)
        _single("points_8000_at_3001", "points", "fp32c", 8000, box, 12, T=3001),
        # a training step of a small system: energy, then dE/dx and dE/dq by autograd
        _single("energy_2000", "energy", "fp32c", 2000, cube, 8, "pm1", terms="fast"),
        # the differentiation workload: 1e5 tight dipoles, refined float32 terms
        _single("energy_dipoles_200000", "energy", "fp32c", 200000, long, 16, "dipoles", terms="refined"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eval32", "eval32", "graph", "fp64", "fp64", "ff", "batch", "points", "energy"])
    d = rng.choice(BOXES)
    p = rng.choice(sorted(PM))
    if kind == "eval32":
        c = _single("", "eval", "fp32c", _log_int(rng, 500, 100000), d, p)
    elif kind == "graph":
        c = _single("", "graph", "fp32c", _log_int(rng, 500, 6000), d, p)
    elif kind == "fp64":
        if rng.random() < 0.25:               # even lattices of 8^3 to 20^3 ions
            c = _single("", "eval", "fp64", (2 * rng.randint(4, 10)) ** 3, BOXES[0], p, "lattice")
        else:
            c = _single("", rng.choice(["eval", "call"]), "fp64", _log_int(rng, 500, 20000), d, p)
    elif kind == "ff":
        c = _single("", "eval", "ff", _log_int(rng, 500, 40000), d, p)
    elif kind == "batch":
        c = {"api": "batch", "precision": "fp32c", "systems": _log_int(rng, 12, 40), "n_lo": 500, "n_hi": 20000,
             "shape": rng.randint(10, 10 ** 6)}
    elif kind == "points":
        c = _single("", "points", rng.choice(["fp32c", "fp32c", "ff"]), _log_int(rng, 1000, 30000), d, p,
                    T=_log_int(rng, 200, 20000))
    else:
        terms = rng.choice(["fast", "refined"])
        if rng.random() < 0.5:
            c = _single("", "energy", "fp32c", 2 * _log_int(rng, 500, 30000), d, p, "dipoles", terms=terms)
        else:
            c = _single("", "energy", rng.choice(["fp32c", "fp64"]), _log_int(rng, 500, 8000), d, p, terms=terms)
    c.pop("name", None)
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _box(case):
    return (case["d1"], case["d2"], case["d3"])


def _uniform(N, d, gen):
    dd = torch.tensor(d, dtype=torch.float64, device=DEV)
    x = (torch.rand((N, 3), dtype=torch.float64, device=DEV, generator=gen) - 0.5) * dd
    return torch.minimum(x, torch.nextafter(0.5 * dd, torch.zeros_like(dd)))


def _wrap(x, d):
    dd = torch.tensor(d, dtype=torch.float64, device=DEV)
    x = x - dd * torch.floor(x / dd + 0.5)
    return torch.maximum(torch.minimum(x, torch.nextafter(0.5 * dd, torch.zeros_like(dd))), -0.5 * dd)


def _pm1(N, gen):
    q = torch.ones(N, dtype=torch.float64, device=DEV)
    q[torch.randperm(N, device=DEV, generator=gen)[: N // 2]] = -1.0
    return q


def _system(N, d, charges, gen):
    """Positions (N, 3) in [-d/2, d/2) and neutral charges (N) on the device."""
    if charges == "lattice":
        n = round(N ** (1.0 / 3.0))
        k = torch.arange(n, dtype=torch.float64, device=DEV)
        I, J, K = torch.meshgrid(k, k, k, indexing="ij")
        a = d[0] / n
        x = torch.stack([(I + 0.5) * a - 0.5 * d[0], (J + 0.5) * a - 0.5 * d[1], (K + 0.5) * a - 0.5 * d[2]], -1)
        x = x.reshape(-1, 3)
        x = x + 0.05 * a * torch.randn(x.shape, dtype=torch.float64, device=DEV, generator=gen)
        q = (1.0 - 2.0 * ((I + J + K) % 2.0)).reshape(-1).contiguous()
        return _wrap(x, d), q
    if charges == "dipoles":                   # +-0.8 at separation 0.01 about uniform centres
        c = _uniform(N // 2, d, gen)
        e = torch.randn((N // 2, 3), dtype=torch.float64, device=DEV, generator=gen)
        e = 0.005 * d[0] * e / e.norm(dim=1, keepdim=True)
        x = torch.stack([_wrap(c + e, d), _wrap(c - e, d)], 1).reshape(-1, 3).contiguous()
        q = torch.tensor([0.8, -0.8], dtype=torch.float64, device=DEV).repeat(N // 2)
        return x, q
    x = _uniform(N, d, gen)
    if charges == "pm1":
        return x, _pm1(N, gen)
    q = torch.randn(N, dtype=torch.float64, device=DEV, generator=gen)
    return x, q - q.mean()


def _batch_systems(case):
    """Sizes, boxes, degrees and near blocks as the batch workload draws them."""
    rng = np.random.default_rng(case["shape"])
    out = []
    for _ in range(case["systems"]):
        N = int(math.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]))))
        N -= N % 2
        d = (1.0, float(rng.uniform(1.0, 2.0)), float(rng.uniform(1.0, 2.0)))
        p, M = W.BATCH_PM[int(rng.integers(0, len(W.BATCH_PM)))]
        out.append(types.SimpleNamespace(N=N, d=d, p=p, M=M, K=W.batch_near_block(d)))
    return out


def _inputs(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    if case["api"] == "batch":
        parts = [_system(s.N, s.d, "pm1", gen) for s in _batch_systems(case)]
        return torch.cat([x for x, _ in parts]), torch.cat([q for _, q in parts])
    x, q = _system(case["N"], _box(case), case["charges"], gen)
    y = _uniform(case["T"], _box(case), gen) if case["api"] == "points" else None
    return x, q, y


def prepare(case, seed):
    s = types.SimpleNamespace(api=case["api"])
    if s.api == "batch":
        s.x, s.q = _inputs(case, seed)
        s.handle = B.PeriodicBatch(_batch_systems(case), precision=case["precision"])
        s.phi = torch.empty_like(s.q)
        s.grad = torch.empty_like(s.x)
        return s
    s.x, s.q, s.y = _inputs(case, seed)
    if s.api == "energy":
        s.handle = PeriodicCoulombEnergy(_box(case), case["p"], case["M"], precision=case["precision"],
                                         terms=case["terms"])
        s.x.requires_grad_(True)
        s.q.requires_grad_(True)
        return s
    s.handle = B.PeriodicCoulomb(_box(case), case["p"], case["M"], precision=case["precision"])
    n = s.y.shape[0] if s.api == "points" else s.q.numel()
    s.phi = torch.empty(n, dtype=torch.float64, device=DEV)
    s.grad = torch.empty((n, 3), dtype=torch.float64, device=DEV)
    return s


def run(s):
    if s.api == "call":
        phi, grad = s.handle(s.x, s.q)
        return {"phi": phi, "grad": grad}
    if s.api == "energy":
        E = s.handle(s.x, s.q)
        dEdx, dEdq = torch.autograd.grad(E, (s.x, s.q))
        return {"E": E.detach(), "dEdx": dEdx, "dEdq": dEdq}
    if s.api == "batch":
        B.psum_batch_eval(s.handle.batch, s.x, s.q, s.phi, s.grad, use_graph=True)
    elif s.api == "graph":
        B.psum_eval_graph(s.handle.plan, s.x, s.q, s.phi, s.grad)
    elif s.api == "points":
        B.psum_eval_points(s.handle.plan, s.x, s.q, s.y, s.phi, s.grad)
    else:
        B.psum_eval(s.handle.plan, s.x, s.q, s.phi, s.grad)
    return {"phi": s.phi, "grad": s.grad}


def work(case):
    """Bytes: charges in, results out.  Operations: 14 per (target, source, image) term of potential
    and field, 9 per term of the potential alone, each check point with the images of its two
    layers, and about 12 per (target, expansion term); the derivatives add the check points'
    potential and field at the charges and one more expansion."""
    if case["api"] == "batch":
        b = f = 0.0
        for s in _batch_systems(case):
            n_img = math.prod(2 * k + 1 for k in s.K)
            b += 64.0 * s.N
            f += 14.0 * n_img * s.N * s.N + 9.0 * 18 * s.N * s.M + 12.0 * (s.p + 1) ** 2 * s.N
        return {"bytes": b, "flops": f}
    N, M, P = case["N"], case["M"], (case["p"] + 1) ** 2
    T = case.get("T", N)
    b = 32.0 * N + 32.0 * T + (24.0 * T if case["api"] == "points" else 0.0)
    f = 14.0 * 27 * N * T + 9.0 * 18 * N * M + 12.0 * P * T
    if case["api"] == "energy":
        f += 14.0 * 18 * N * M + 12.0 * P * N
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# the same results in plain float64
# ---------------------------------------------------------------------------
def _harmonics(u, p, grad):
    """Renormalised regular solid harmonics (P, n) at u (n, 3) and their derivatives (P, 3, n)."""
    x, y, z = (u[:, k] for k in range(3))
    r2 = x * x + y * y + z * z
    n_pts, P = u.shape[0], (p + 1) ** 2
    R = torch.zeros((P, n_pts), dtype=torch.float64, device=u.device)
    G = torch.zeros((P, 3, n_pts), dtype=torch.float64, device=u.device) if grad else None
    eye = torch.eye(3, dtype=torch.float64, device=u.device)[:, :, None]
    at = lambda n, m: n * (n + 1) + m                                             # noqa: E731
    R[0] = 1.0
    for m in range(1, p + 1):
        c = math.sqrt((2 * m - 1) / (2 * m))
        i, j, a = at(m, m), at(m, -m), at(m - 1, m - 1)
        b = at(m - 1, 1 - m)
        Rb = R[b] if m > 1 else torch.zeros_like(x)
        R[i], R[j] = -c * (x * R[a] + y * Rb), c * (y * R[a] - x * Rb)
        if grad:
            Gb = G[b] if m > 1 else torch.zeros_like(G[a])
            G[i] = -c * (eye[0] * R[a] + x * G[a] + eye[1] * Rb + y * Gb)
            G[j] = c * (eye[1] * R[a] + y * G[a] - eye[0] * Rb - x * Gb)
    for m in range(-p, p + 1):
        k = abs(m)
        for n in range(k + 1, p + 1):
            den = math.sqrt((n - k) * (n + k))
            e1, e2 = (2 * n - 1) / den, math.sqrt((n - k - 1) * (n + k - 1)) / den
            i, a, b = at(n, m), at(n - 1, m), at(n - 2, m) if n > k + 1 else at(n - 1, m)
            R[i] = -e1 * z * R[a] - e2 * r2 * R[b]
            if grad:
                G[i] = -e1 * (eye[2] * R[a] + z * G[a]) - e2 * (2.0 * u.T * R[b] + r2 * G[b])
    return R, G


def _near(t, x, q, d, K, grad, Rt=None):
    """Direct image sum of the charges (x, q) at t: potential and field, K(0) = 0."""
    phi = torch.zeros(t.shape[0], dtype=torch.float64, device=t.device)
    g = torch.zeros((t.shape[0], 3), dtype=torch.float64, device=t.device) if grad else None
    step = max(1, (1 << 26) // max(1, x.shape[0]))
    shifts = [(i * d[0], j * d[1], k * d[2]) for i in range(-K[0], K[0] + 1) for j in range(-K[1], K[1] + 1)
              for k in range(-K[2], K[2] + 1)]
    for a in range(0, t.shape[0], step):
        tt = t[a:a + step]
        for s in shifts:
            e = [x[None, :, k] - (tt[:, k, None] - s[k]) for k in range(3)]
            r2 = e[0] * e[0] + e[1] * e[1] + e[2] * e[2]
            ri = torch.where(r2 > 0, r2, torch.ones_like(r2)).sqrt_().reciprocal_()
            ri = torch.where(r2 > 0, ri, torch.zeros_like(ri))
            phi[a:a + step] += ri @ q
            if grad:
                w = ri * ri * ri * q[None, :]
                for k in range(3):
                    g[a:a + step, k] += (w * e[k]).sum(1)
    return phi, g


def _prism(x, H):
    """Newtonian potential of the uniform box [-H, H] at points inside it: the 8-corner sum."""
    U = torch.zeros(x.shape[0], dtype=torch.float64, device=x.device)
    for c in range(8):
        s = [1.0 if c >> k & 1 else -1.0 for k in range(3)]
        v = [s[k] * H[k] - x[:, k] for k in range(3)]
        r = (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]).sqrt()
        F = torch.zeros_like(U)
        for k in range(3):
            a, b, e = v[k], v[(k + 1) % 3], v[(k + 2) % 3]
            lg = torch.where(e >= 0, (e + r).log(), ((a * a + b * b) / (r - e)).log())
            F += a * b * lg - 0.5 * a * a * torch.atan(b * e / (a * r))
        U += s[0] * s[1] * s[2] * F
    return U


def _exact_system(x, q, d, p, M, K, y=None, energy=False):
    R0 = 0.5 * math.sqrt(sum(v * v for v in d))
    l = np.arange(M, dtype=np.float64)
    cz = 1.0 - (2.0 * l + 1.0) / M
    rho, az = np.sqrt(1.0 - cz * cz), l * math.pi * (3.0 - math.sqrt(5.0))
    Y = R0 * np.stack([rho * np.cos(az), rho * np.sin(az), cz], 1)
    k = np.argmax(np.abs(Y) / np.asarray(d), axis=1)
    Yt = Y.copy()
    rows = np.arange(M)
    Yt[rows, k] -= np.sign(Y[rows, k]) * np.asarray(d)[k]
    Y, Yt = torch.from_numpy(Y).to(x.device), torch.from_numpy(Yt).to(x.device)
    A = (_harmonics(Y / R0, p, False)[0] - _harmonics(Yt / R0, p, False)[0])[1:].T.cpu().numpy()
    f = (_near(Yt, x, q, d, K, False)[0] - _near(Y, x, q, d, K, False)[0]).cpu().numpy()
    U, S, Vt = np.linalg.svd(A, full_matrices=False)
    C = np.zeros((p + 1) ** 2)
    C[1:] = Vt.T @ ((U.T @ f) / S)
    nodes, wts = np.polynomial.legendre.leggauss(p // 2 + 1)
    g3 = np.stack(np.meshgrid(*(0.5 * v * nodes for v in d), indexing="ij"), -1).reshape(-1, 3)
    w3 = np.einsum("i,j,k->ijk", wts, wts, wts).reshape(-1) / 8.0
    Rbox = _harmonics(torch.from_numpy(g3 / R0), p, False)[0].numpy() @ w3
    H = [0.5 * (2 * K[i] + 1) * d[i] for i in range(3)]
    C[0] = -float((q * _prism(x, H)).sum()) / (d[0] * d[1] * d[2]) - float(C[1:] @ Rbox[1:])
    Ct = torch.from_numpy(C).to(x.device)
    t = x if y is None else y
    phi_n, g_n = _near(t, x, q, d, K, True)
    R, G = _harmonics(t / R0, p, True)
    phi_f, g_f = Ct @ R, torch.einsum("t,tkn->nk", Ct, G) / R0
    if not energy:
        return {"phi": phi_n + phi_f, "grad": g_n + g_f}
    w = (R[1:] @ q).cpu().numpy()
    u = torch.from_numpy(U @ ((Vt @ w) / S)).to(x.device)
    psi, gpsi = _near(x, torch.cat([Yt, Y]), torch.cat([u, -u]), d, K, True)
    return {"E": 0.5 * (q * (phi_n + phi_f)).sum(), "dEdx": q[:, None] * (g_n + 0.5 * g_f + 0.5 * gpsi),
            "dEdq": phi_n + 0.5 * phi_f + 0.5 * psi}


def exact(case, seed):
    if case["api"] == "batch":
        systems = _batch_systems(case)
        if sum(s.N * s.N for s in systems) > 6e8:
            return None
        x, q = _inputs(case, seed)
        out, n0 = [], 0
        for s in systems:
            out.append(_exact_system(x[n0:n0 + s.N], q[n0:n0 + s.N], s.d, s.p, s.M, s.K))
            n0 += s.N
        return {k: torch.cat([o[k] for o in out]) for k in ("phi", "grad")}
    if case["N"] * case.get("T", case["N"]) > 6e8:
        return None
    x, q, y = _inputs(case, seed)
    return _exact_system(x, q, _box(case), case["p"], case["M"], (1, 1, 1), y, case["api"] == "energy")
