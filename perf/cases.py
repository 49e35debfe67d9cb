"""Performance cases: what users of this framework have it compute, through its public entry points.

Sizes are those of the repository's own configurations (the deterministic 32^3 validation run, the
64^3 x 64 benchmark ensemble, the 128^3 x 32 target shape, the three-level viscosity batch, the
64^3 x 16 adjoint, the M = 100 Wasserstein comparison) or generic ones between them.

Kinds of cases:
  run    - one Monte Carlo job: initialise M samples from their parameters, advance them, read the
           energy and the mean / variance fields (M = 1: the density and velocity fields);
  levels - the same for a viscosity sequence of three resolutions advanced together;
  grad   - J and dJ/dX of every sample, forward and backward through the autograd function;
  stats  - the spectral and structure-function statistics of a snapshot;
  w1     - one- and two-point Wasserstein distances between two ensembles.
"""
import itertools
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2608_23786_gb300 import Ensemble, mclbm
from paper_2608_23786_gb300.autograd import ensemble_objective

ELEM = {"fp64": 8, "fp32": 4, "fp16": 2}


def _run(name, N, M, prec, pattern, steps, lattice=19, gamma=False):
    c = {"kind": "run", "N": N, "M": M, "prec": prec, "pattern": pattern, "steps": steps, "lattice": lattice,
         "exact_gamma": gamma}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one sample in the plain FP64 method: the validation run against the deterministic vortex
        _run("run32_m1_fp64", 32, 1, "fp64", "pull", 200),
        # a small ensemble on the coarsest lattice of a convergence study, an odd number of samples
        _run("run32_m7_fp32", 32, 7, "fp32", "pull", 200),
        # the benchmark ensemble, end to end
        _run("run64_m64_fp32", 64, 64, "fp32", "pull", 50),
        # the target shape in the in-place streaming pattern, an odd number of steps
        _run("run128_m32_fp32_aa", 128, 32, "fp32", "aa", 21),
        # the fine level of a viscosity sequence in half-precision storage
        _run("run256_m8_fp16_aa", 256, 8, "fp16", "aa", 10),
        # the 27-velocity lattice
        _run("run64_m16_q27_fp32", 64, 16, "fp32", "pull", 50, lattice=27),
        # a reference ensemble in FP64, against which reduced storage is judged
        _run("run64_m8_fp64", 64, 8, "fp64", "pull", 20),
        # the exact entropic stabiliser instead of its closed form
        _run("run64_m8_fp32_gamma", 64, 8, "fp32", "pull", 20, gamma=True),
        # three viscosity levels, 1 : 4 : 16 steps per macro step, advanced as one batch
        {"name": "levels3_fp16_aa", "kind": "levels", "N": 64, "M": 64, "prec": "fp16", "pattern": "aa", "macro": 2},
        # gradient of every sample's final energy with respect to its 24 parameters
        {"name": "grad64_m16_fp32", "kind": "grad", "N": 64, "M": 16, "prec": "fp32", "steps": 100, "ckpt": 50,
         "objective": "energy"},
        # the statistics of one snapshot: shell spectrum, S_2 from the autocorrelation, S_p along axes
        {"name": "stats128_m4_fp32", "kind": "stats", "N": 128, "M": 4, "prec": "fp32", "pmax": 6},
        # one-point and two-point W1 between two ensembles of 100 samples on the 8^3 grid
        {"name": "w1_32_m100", "kind": "w1", "N": 32, "M": 100, "MB": 100, "points": 8, "vector": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# seconds of one node update, roughly, for bounding what draw() asks for
_UPDATE_S = {"fp64": 1e-9, "fp32": 2.5e-11, "fp16": 1.4e-11}


def draw(rng):
    kind = rng.choices(["run", "levels", "grad", "stats", "w1"], [12, 1, 2, 2, 1])[0]
    if kind == "run":
        prec = rng.choices(["fp32", "fp16", "fp64"], [4, 3, 2])[0]
        pattern = rng.choice(["pull", "aa"])
        lattice = rng.choices([19, 27], [4, 1])[0]
        gamma = rng.random() < 0.08
        N = 2 ** rng.randint(3, 8 if prec != "fp64" and not gamma else 6)
        nodes = min(1 << 27, int(6e10 / (2 * lattice * ELEM[prec]))) if prec != "fp64" else 1 << 21
        M = min(200, _log_int(rng, 1, max(1, min(nodes, nodes >> (3 if gamma else 0)) // N**3)))
        cost = M * N**3 * _UPDATE_S[prec] * (6 if gamma else 1) * lattice / 19
        steps = _log_int(rng, 3, max(3, min(400, int(0.06 / cost))))
        return _run(None, N, M, prec, pattern, steps, lattice, gamma)
    prec = rng.choice(["fp32", "fp16"])
    if kind == "levels":
        return {"kind": "levels", "N": 2 ** rng.randint(4, 6), "M": 4 * _log_int(rng, 1, 16), "prec": prec,
                "pattern": rng.choice(["pull", "aa"]), "macro": rng.randint(1, 3)}
    if kind == "grad":
        N = 2 ** rng.randint(4, 6)
        M = _log_int(rng, 1, min(64, (1 << 22) // N**3))
        return {"kind": "grad", "N": N, "M": M, "prec": prec, "steps": _log_int(rng, 20, 100),
                "ckpt": _log_int(rng, 10, 50), "objective": rng.choice(["energy", "enstrophy"])}
    if kind == "stats":
        N = 2 ** rng.randint(4, 7)
        return {"kind": "stats", "N": N, "M": _log_int(rng, 1, min(32, (1 << 23) // N**3)), "prec": prec,
                "pmax": rng.randint(2, 6)}
    M = _log_int(rng, 4, 100)
    return {"kind": "w1", "N": 2 ** rng.randint(4, 5), "M": M, "MB": rng.choice([M, max(2, M // 2)]),
            "points": rng.choice([4, 8]), "vector": rng.random() < 0.75}


# ---- what a program has in hand, and the call -----------------------------------------------------


def _physics(N):
    """Reynolds and Mach number of a lattice, as in the configurations (64^3: 800, 0.025)."""
    return {"Re": 12.5 * N, "Ma": 1.6 / max(N, 32)}


def _params(seed, M, k=0):
    """[M][24] uniform parameters of the randomized Taylor-Green samples."""
    return np.random.default_rng([int(seed), k]).uniform(-0.025, 0.025, (M, 24))


def _levels(c):
    """(N, M, steps per macro step) of the three levels."""
    return [(c["N"], c["M"], 1), (2 * c["N"], c["M"] // 2, 4), (4 * c["N"], c["M"] // 8 or 2, 16)]


class _Levels:
    """The contexts of a viscosity sequence and the batch that advances them."""

    def __init__(self, c, seed):
        self.stream = torch.cuda.Stream()
        spec = _levels(c)
        self.ens = [Ensemble(N, M, precision=c["prec"], pattern=c["pattern"], stream=self.stream, **_physics(N))
                    for N, M, _ in spec]
        self.X = [_params(seed, M, k) for k, (_, M, _) in enumerate(spec)]
        self.batch = mclbm.mclbm_batch_create([e.ctx for e in self.ens], [s for _, _, s in spec])

    def __del__(self):
        if getattr(self, "batch", None) is not None:
            mclbm.mclbm_batch_destroy(self.batch)


SNAPSHOT_STEPS = 10  # steps before the statistics of a snapshot


def prepare(case, seed):
    c = case
    if c["kind"] == "run":
        ens = Ensemble(c["N"], c["M"], precision=c["prec"], pattern=c["pattern"], lattice=c["lattice"],
                       exact_gamma=c["exact_gamma"], **_physics(c["N"]))
        return {"case": c, "ens": ens, "X": _params(seed, c["M"])}
    if c["kind"] == "levels":
        return {"case": c, "levels": _Levels(c, seed)}
    if c["kind"] == "grad":
        return {"case": c, "X": torch.from_numpy(_params(seed, c["M"]))}
    if c["kind"] == "stats":
        ens = Ensemble(c["N"], c["M"], precision=c["prec"], **_physics(c["N"]))
        return {"case": c, "ens": ens.init(_params(seed, c["M"])).step(SNAPSHOT_STEPS)}
    a, b = (Ensemble(c["N"], M, precision="fp32", **_physics(c["N"])).init(_params(seed, M, k)).step(SNAPSHOT_STEPS)
            for k, M in enumerate((c["M"], c["MB"])))
    return {"case": c, "a": a, "b": b}


def _snapshot(ens):
    if ens.M == 1:
        rho, u = ens.moments(0)
        return {"rho": rho, "u": u}
    E, mean, var = ens.energy_mean_var()
    return {"E": E, "mean": mean, "var": var}


def run(state):
    c = state["case"]
    if c["kind"] == "run":
        return _snapshot(state["ens"].init(state["X"]).step(c["steps"]))
    if c["kind"] == "levels":
        lv = state["levels"]
        for ens, X in zip(lv.ens, lv.X):
            ens.init(X)
        mclbm.mclbm_batch_step(lv.batch, c["macro"])
        return [_snapshot(ens) for ens in lv.ens]
    if c["kind"] == "grad":
        X = state["X"].clone().requires_grad_(True)
        J = ensemble_objective(X, c["N"], nsteps=c["steps"], ckpt_every=c["ckpt"], objective=c["objective"],
                               precision=c["prec"], **_physics(c["N"]))
        J.sum().backward()
        return {"J": J.detach(), "grad": X.grad}
    if c["kind"] == "stats":
        ens = state["ens"]
        return {"spectrum": ens.spectrum(), "S2": ens.sf_trace(), "Sp": ens.sf_axes(c["pmax"])}
    a, b, Q = state["a"], state["b"], c["points"]
    W, per_point = a.w1(b, Q, per_point=True)
    return {"w1": W, "w1_points": per_point, "w1_2pt": a.w1_2pt(b, Q, vector=c["vector"])}


# ---- what a pass cannot do without ----------------------------------------------------------------


def _state(N, M, prec, lattice=19):
    return M * N**3 * lattice * ELEM[prec]


def _fields(N, M):
    return N**3 * 8 * (4 if M == 1 else 6)


def _update_flops(lattice, gamma=False):
    """Operations of one node update: about 15 per population (an exact stabiliser takes a logarithm,
    a quotient and six more operations per population and evaluation, and at least two evaluations)."""
    return lattice * (15 + (2 * 30 if gamma else 0))


def work(case):
    """Bytes: the state written once and read once (it does not fit on the chip), and the results.  Flops:
    the operations of the method."""
    c = case
    N, M = c["N"], c["M"]
    if c["kind"] == "run":
        return {"bytes": 2 * _state(N, M, c["prec"], c["lattice"]) + _fields(N, M),
                "flops": M * N**3 * c["steps"] * _update_flops(c["lattice"], c["exact_gamma"])}
    if c["kind"] == "levels":
        spec = _levels(c)
        return {"bytes": sum(2 * _state(n, m, c["prec"]) + _fields(n, m) for n, m, _ in spec),
                "flops": sum(m * n**3 * s for n, m, s in spec) * c["macro"] * _update_flops(19)}
    if c["kind"] == "grad":
        # the forward states that the reverse sweep reads are written once and read once; the product
        # with the transposed Jacobian takes about three times a collision
        return {"bytes": 2 * c["steps"] * _state(N, M, c["prec"]),
                "flops": M * N**3 * c["steps"] * 4 * _update_flops(19)}
    if c["kind"] == "stats":
        n = N**3
        fft = 5 * n * math.log2(n)
        # three real fields forward and one autocorrelation back at half a complex transform each, for
        # each of the two spectral statistics; 1.5 N differences of pmax + 2 operations per node
        return {"bytes": _state(N, M, c["prec"]), "flops": M * (1.5 * fft + 2 * fft + n * 1.5 * N * (c["pmax"] + 2))}
    G = c["points"] ** 3
    pairs, K = G * (G + 1) // 2, 6 if c["vector"] else 2
    # the cost matrix of every pair's transport problem, once
    return {"bytes": (M + c["MB"]) * G * 24,
            "flops": pairs * (1 if c["vector"] else 3) * M * c["MB"] * (3 * K + 1)}


# ---- the same in 64 bits, plainly -----------------------------------------------------------------

_MOST_UPDATES = {19: 3.2e9, 27: 2.2e9}  # node updates that plain torch does in some seconds on a GPU


class _Lattice:
    """Velocities, weights and the moment matrices of a velocity set, and one sample's KBC update."""

    def __init__(self, Q, device):
        self.c = [c for c in itertools.product((-1, 0, 1), repeat=3) if Q == 27 or sum(map(abs, c)) < 3]
        table = {19: (1 / 3, 1 / 18, 1 / 36), 27: (8 / 27, 2 / 27, 1 / 54, 1 / 216)}[Q]
        kw = {"dtype": torch.float64, "device": device}
        self.w = torch.tensor([table[sum(map(abs, c))] for c in self.c], **kw)
        c = torch.tensor(self.c, **kw)
        self.cT = c.T.contiguous()  # [3][Q]
        self.cm = c
        # second moments xx, yy, zz, xy, xz, yz of the populations, and the shear part that carries a
        # given deviatoric tensor: D_aa / 2 on the faces, s l P_ab / 4 on the edges
        ab = [(0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)]
        self.P = torch.stack([c[:, a] * c[:, b] for a, b in ab])
        n2 = (c * c).sum(1)
        share = [(c[:, a] * c[:, b]) * ((n2 == 1) * 0.5 if a == b else (n2 == 2) * 0.25) for a, b in ab]
        self.S = torch.stack(share, 1).contiguous()  # [Q][6]

    def equilibrium(self, rho, u):
        cu = self.cm @ u
        return self.w[:, None] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (u * u).sum(0))

    def moments(self, f):
        rho = f.sum(0)
        return rho, (self.cT @ f) / rho

    def collide(self, f, omega, exact_gamma):
        feq = self.equilibrium(*self.moments(f))
        fneq = f - feq
        D = self.P @ fneq
        D = torch.cat([D[:3] - D[:3].mean(0), D[3:]])
        ds = self.S @ D
        dh = fneq - ds
        hw = dh / feq
        sh, hh = (ds * hw).sum(0), (dh * hw).sum(0)
        zero = hh == 0
        gamma = 2 / omega - (2 - 2 / omega) * sh / torch.where(zero, torch.ones_like(hh), hh)
        if exact_gamma:
            gamma = self.minimiser(f - omega * ds, 0.5 * omega * dh, omega, gamma)
        gamma = torch.where(zero, torch.full_like(gamma, 2.0), gamma)
        return f - omega * ds - 0.5 * omega * gamma * dh

    def minimiser(self, a, b, omega, closed):
        """The g in [0, 4 / omega] at which sum f* ln(f* / w), f* = a - g b, is least: bisection."""
        r = a / b
        hi = torch.where(b > 0, r, torch.full_like(r, 4 / omega)).amin(0).clamp(max=4 / omega)
        lo = torch.where(b < 0, r, torch.zeros_like(r)).amax(0).clamp(min=0)
        ok = lo < hi
        am1, bw = a / self.w[:, None] - 1, b / self.w[:, None]
        for _ in range(44):
            mid = 0.5 * (lo + hi)
            up = (b * torch.log1p(am1 - mid * bw)).sum(0) > 0
            lo, hi = torch.where(up, mid, lo), torch.where(up, hi, mid)
        return torch.where(ok, 0.5 * (lo + hi), closed)

    def step(self, f, N, omega, exact_gamma=False):
        post = self.collide(f, omega, exact_gamma).view(-1, N, N, N)
        return torch.stack([torch.roll(p, (z, y, x), (0, 1, 2)) for p, (x, y, z) in zip(post, self.c)]).view(len(self.c), -1)


def _units(N):
    p = _physics(N)
    u_lat, dx = p["Ma"] / math.sqrt(3), 2 * math.pi / N
    nu_lat = (1 / p["Re"]) * (u_lat * dx) / dx**2
    return u_lat, 1 / (3 * nu_lat + 0.5)


def _initial(lat, N, X, u_lat):
    """f [Q][N^3] of one sample, X [24] (a tensor)."""
    x = torch.arange(N, dtype=torch.float64, device=X.device) * (2 * math.pi / N)
    s, co = torch.sin(x), torch.cos(x)
    A = torch.stack([torch.sin(2 * x), torch.cos(2 * x)])
    pert = torch.einsum("aijk,ix,jy,kz->azyx", X.view(3, 2, 2, 2), A, A, A) / 8
    ux = co[:, None, None] * co[None, :, None] * s[None, None, :]
    uy = -co[:, None, None] * s[None, :, None] * co[None, None, :]
    u = u_lat * (torch.stack([ux, uy, torch.zeros_like(ux)]) + pert)
    return lat.equilibrium(torch.ones(N**3, dtype=torch.float64, device=X.device), u.reshape(3, -1))


def _advance(N, X, steps, lattice=19, exact_gamma=False):
    """(rho [N^3], u [3][N^3]) of one sample after `steps` steps."""
    lat = _Lattice(lattice, X.device)
    u_lat, omega = _units(N)
    f = _initial(lat, N, X, u_lat)
    for _ in range(steps):
        f = lat.step(f, N, omega, exact_gamma)
    rho, u = lat.moments(f)
    return rho, u / u_lat


def _exact_snapshot(N, X, steps, lattice=19, exact_gamma=False):
    E, total, square, first = [], 0, 0, None
    M = len(X)
    for m in range(M):
        rho, u = _advance(N, X[m], steps, lattice, exact_gamma)
        if M == 1:
            return {"rho": rho.view(N, N, N), "u": u.view(3, N, N, N)}
        first = u if first is None else first
        E.append(0.5 * float((u * u).sum()) / N**3)
        d = u - first
        total, square = total + d, square + d * d
    mean, var = first + total / M, (square - total * total / M) / (M - 1)
    return {"E": np.array(E), "mean": mean.view(3, N, N, N), "var": var.view(3, N, N, N)}


def _exact_stats(N, X, pmax):
    k = torch.fft.fftfreq(N, 1 / N, device=X.device).to(torch.float64)
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :] ** 2
    shell = torch.round(torch.sqrt(k2)).long().flatten()
    count = torch.bincount(shell)[: N // 2 + 1].double()

    def shells(v):
        return torch.bincount(shell, v.flatten())[: N // 2 + 1] / count

    out = {"spectrum": [], "S2": [], "Sp": []}
    for x in X:
        u = _advance(N, x, SNAPSHOT_STEPS)[1].view(3, N, N, N)
        power = sum((t * t.conj()).real for t in (torch.fft.fftn(v) for v in u))
        out["spectrum"].append(4 * math.pi * shells(0.5 * k2 * power / N**6))
        R = torch.fft.ifftn(power).real / N**3
        out["S2"].append(shells(2 * (R[0, 0, 0] - R)))
        S = torch.zeros((pmax - 1, N // 2), dtype=torch.float64)
        for r in range(1, N // 2 + 1):
            d = torch.stack([(torch.roll(u[a], -r, 2 - a) - u[a]).abs() for a in range(3)])
            for p in range(2, pmax + 1):
                S[p - 2, r - 1] = float((d**p).sum()) / (3 * N**3)
        out["Sp"].append(S)
    return {n: torch.stack(v).cpu().numpy() for n, v in out.items()}


def _exact_w1(c, XA, XB):
    N, Q = c["N"], c["points"]
    ua, ub = (torch.stack([_advance(N, x, SNAPSHOT_STEPS)[1].view(3, N, N, N)[:, :: N // Q, :: N // Q, :: N // Q].reshape(3, -1).T
                           for x in X]) for X in (XA, XB))
    # L1 distance of the empirical distribution functions over the merged support
    both = torch.cat([ua, ub]).sort(0)
    sign = torch.cat([torch.full((len(ua),), 1 / len(ua)), torch.full((len(ub),), -1 / len(ub))]).to(ua)
    gap = sign[both.indices].cumsum(0)[:-1].abs()
    per = (gap * both.values.diff(dim=0)).sum(0)
    return {"w1": float(per.sum()) / Q**3, "w1_points": per.cpu().numpy(), "w1_2pt": None}


def _exact_gradient(c, X):
    N = c["N"]
    lat = _Lattice(19, X.device)
    u_lat, omega = _units(N)
    J, G = [], []
    for m in range(len(X)):
        x = X[m].clone().requires_grad_(True)
        f = _initial(lat, N, x, u_lat)
        for _ in range(c["steps"]):
            f = checkpoint(lat.step, f, N, omega, use_reentrant=False)
        u = (lat.moments(f)[1] / u_lat).view(3, N, N, N)
        if c["objective"] == "energy":
            j = 0.5 * (u * u).sum() / N**3
        else:
            def d(v, axis):
                return (torch.roll(v, -1, 2 - axis) - torch.roll(v, 1, 2 - axis)) / (4 * math.pi / N)
            w = (d(u[2], 1) - d(u[1], 2), d(u[0], 2) - d(u[2], 0), d(u[1], 0) - d(u[0], 1))
            j = 0.5 * sum((v * v).sum() for v in w) / N**3
        G.append(torch.autograd.grad(j, x)[0])
        J.append(j.detach())
    return {"J": torch.stack(J).cpu(), "grad": torch.stack(G).cpu()}


def exact(case, seed):
    c = case
    device = "cuda" if torch.cuda.is_available() else "cpu"

    def params(M, k=0):
        return torch.from_numpy(_params(seed, M, k)).to(device)

    N, M = c["N"], c["M"]
    if c["kind"] == "run":
        most = _MOST_UPDATES[c["lattice"]] / (40 if c["exact_gamma"] else 1)
        if M * N**3 * c["steps"] > most:
            return None
        return _exact_snapshot(N, params(M), c["steps"], c["lattice"], c["exact_gamma"])
    if c["kind"] == "levels":
        spec = _levels(c)
        if sum(n**3 * m * s for n, m, s in spec) * c["macro"] > _MOST_UPDATES[19]:
            return None
        return [_exact_snapshot(n, params(m, k), s * c["macro"]) for k, (n, m, s) in enumerate(spec)]
    if c["kind"] == "grad":
        return _exact_gradient(c, params(M))
    if c["kind"] == "stats":
        return _exact_stats(N, params(M), c["pmax"])
    return _exact_w1(c, params(M), params(c["MB"], 1))
