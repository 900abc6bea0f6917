"""What the library is measured on: the calls that a program with particles in a fluctuating channel flow makes.

Every case goes through the public entry points of ``paper_1003_2680_gb300.selm`` with the options and the
sizes that the repository's own workloads use: the uniform channel (2-D and 3-D, with and without the MAC
projection), the refined-patch composite grid, the staggered composite grid, batches of uneven systems and the
exact Stokes mobility.  Inputs are drawn from the seed alone: positions uniform in the box and a few cells off
the walls, N(0, 1) forces and fields.

Time steps: dt = 0.02 h^2 (h the finest spacing) moves a particle by a fraction of a cell per step, as an
Euler-Maruyama step has to.
"""

import math

import numpy as np
import torch

from paper_1003_2680_gb300 import selm as S

_PRECISION = {"fp64": S.SELM_FP64, "fp32": S.SELM_FP32_REFINE64}


def listed():
    return [
        # one chain of a small 2-D channel in FP64: the plain method's own configuration (64^2, six levels),
        # where only latency counts
        {"name": "chain-2d-64-fp64", "kind": "chain", "dim": 2, "n": 64, "levels": 6, "precision": "fp64",
         "particles": 16, "cycles": 4},
        # one stochastic V-cycle on a level field of a small, odd-sized 3-D channel: the sampler's building block
        {"name": "vcycle-48-fp32", "kind": "vcycle", "dim": 3, "n": 48, "precision": "fp32"},
        # a served 2-D request: one Euler-Maruyama step of a wide channel
        {"name": "step-2d-768", "kind": "step", "dim": 2, "n": 768, "precision": "fp32", "projection": False,
         "particles": 600, "cycles": 2},
        # the headline: one Euler-Maruyama step of the 128^3 channel with the MAC projection
        {"name": "step-128-mac", "kind": "step", "dim": 3, "n": 128, "precision": "fp32", "projection": True,
         "particles": 1024, "cycles": 2},
        # the mobility of a set of particles on a grid whose edge is not a power of two (pressure by V-cycles)
        {"name": "mobility-96-mac", "kind": "mobility", "dim": 3, "n": 96, "precision": "fp32", "projection": True,
         "particles": 700},
        # the largest served request: one step of the 192^3 channel
        {"name": "step-192", "kind": "step", "dim": 3, "n": 192, "precision": "fp32", "projection": False,
         "particles": 4096, "cycles": 2},
        # thermal samples of the composite grid at its benchmark size (about 1e8 unknowns)
        {"name": "composite-sample-256", "kind": "comp_sample", "dim": 3, "n": 256, "K": 32, "ncomp": 3,
         "precision": "fp32", "cycles": 2},
        # one scalar solve on a smaller composite grid with odd coarse levels and an odd patch, all in FP64
        {"name": "composite-solve-80-fp64", "kind": "comp_solve", "dim": 3, "n": 80, "K": 9, "ncomp": 1,
         "precision": "fp64"},
        # one step of the staggered composite grid with its projections
        {"name": "mac-step-64", "kind": "mac_step", "dim": 3, "n": 64, "K": 8, "precision": "fp32",
         "projection": True, "particles": 1000, "cycles": 2},
        # thermal samples of a small staggered composite grid in FP64
        {"name": "mac-sample-32-fp64", "kind": "mac_sample", "dim": 3, "n": 32, "K": 5, "precision": "fp64",
         "cycles": 2},
        # uneven systems advanced together
        {"name": "batch-16", "kind": "batch", "systems": 16, "mix": 0, "cycles": 2},
        # the exact Stokes mobility of a set of particles
        {"name": "stokes-mobility-64", "kind": "stokes", "dim": 3, "n": 64, "precision": "fp32", "particles": 256},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["chain", "vcycle", "step2", "step3", "mobility", "comp_sample", "comp_solve", "mac_step",
                       "mac_sample", "batch", "stokes"])
    precision = rng.choice(["fp32", "fp32", "fp64"])
    if kind == "chain":
        return {"kind": "chain", "dim": 2, "n": 8 * _log(rng, 4, 40), "levels": 0,
                "precision": rng.choice(["fp64", "fp32"]), "particles": _log(rng, 1, 100), "cycles": rng.randint(1, 8)}
    if kind == "vcycle":
        return {"kind": "vcycle", "dim": 3, "n": 8 * rng.randint(2, 20), "precision": precision}
    if kind == "step2":
        return {"kind": "step", "dim": 2, "n": 16 * _log(rng, 8, 64), "precision": "fp32",
                "projection": rng.random() < 0.3, "particles": _log(rng, 16, 4096), "cycles": rng.randint(1, 3)}
    if kind == "step3":
        return {"kind": "step", "dim": 3, "n": 16 * rng.randint(2, 12), "precision": "fp32",
                "projection": rng.random() < 0.5, "particles": _log(rng, 16, 4096), "cycles": rng.randint(1, 3)}
    if kind == "mobility":
        return {"kind": "mobility", "dim": 3, "n": 16 * rng.randint(2, 8), "precision": precision,
                "projection": rng.random() < 0.5, "particles": _log(rng, 1, 4096)}
    if kind == "comp_sample":
        n = 16 * rng.randint(2, 15)
        return {"kind": "comp_sample", "dim": 3, "n": n, "K": rng.randint(1, n // 8), "ncomp": rng.randint(1, 3),
                "precision": "fp32", "cycles": rng.randint(1, 2)}
    if kind == "comp_solve":
        n = 16 * rng.randint(2, 5)
        return {"kind": "comp_solve", "dim": 3, "n": n, "K": rng.randint(1, min(8, n // 6)),
                "ncomp": 1 if n > 48 else rng.randint(1, 3), "precision": precision}
    if kind == "mac_step":
        n = 8 * rng.randint(2, 6)
        return {"kind": "mac_step", "dim": 3, "n": n, "K": rng.randint(1, n // 6), "precision": precision,
                "projection": rng.random() < 0.7, "particles": _log(rng, 10, 1000), "cycles": rng.randint(1, 3)}
    if kind == "mac_sample":
        n = 8 * rng.randint(2, 6)
        return {"kind": "mac_sample", "dim": 3, "n": n, "K": rng.randint(1, n // 6), "precision": precision,
                "cycles": rng.randint(1, 3)}
    if kind == "batch":
        return {"kind": "batch", "systems": rng.randint(2, 16), "mix": rng.randint(1, 1000), "cycles": 2}
    return {"kind": "stokes", "dim": 3, "n": 16 * rng.randint(2, 4), "precision": "fp32",
            "particles": _log(rng, 1, 256)}


# -- inputs --------------------------------------------------------------------------------------------------
def _particles(count, dim, n, seed):
    rng = np.random.default_rng([seed, 1])
    x = rng.uniform(0.0, 1.0, size=(count, dim))
    x[:, -1] = rng.uniform(2.0 / n, 1.0 - 2.0 / n, size=count)
    return torch.from_numpy(x).cuda()


def _forces(count, dim, seed):
    return torch.from_numpy(np.random.default_rng([seed, 2]).standard_normal((count, dim))).cuda()


def _field(size, seed, dtype):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(size, generator=g, device="cuda", dtype=dtype)


class _Owner:
    """Keeps a handle of the library and gives it back with the state."""

    def __init__(self, handle, destroy):
        self.h, self._destroy = handle, destroy

    def __del__(self):
        torch.cuda.synchronize()
        self._destroy(self.h)


def _mg(case, seed):
    return S.SelmMG(dim=case["dim"], n=case["n"], levels=case.get("levels", 0), kT=1.0,
                    precision=_PRECISION[case["precision"]],
                    projection=S.SELM_PROJ_MAC if case.get("projection") else S.SELM_PROJ_NONE,
                    max_particles=max(1, case.get("particles", 1)), seed=seed, instance=1)


def _mac(case, seed):
    d = S.make_mac_desc(case["dim"], case["n"], case["K"], kT=1.0, precision=_PRECISION[case["precision"]],
                        projection=S.SELM_PROJ_MAC if case.get("projection") else S.SELM_PROJ_NONE, seed=seed,
                        instance=1)
    return _Owner(S.selm_mac_create(d), S.selm_mac_destroy)


def _comp(case, seed):
    d = S.make_comp_desc(case["dim"], case["n"], case["K"], ncomp=case["ncomp"],
                         precision=_PRECISION[case["precision"]], seed=seed, instance=1)
    return _Owner(S.selm_comp_create(d), S.selm_comp_destroy)


def _mix(case):
    """Edges, particle counts and kT of a batch's systems."""
    rng = np.random.default_rng([case["mix"], 3])
    edges = [int(e) for e in rng.choice([32, 48, 64, 96, 128], size=case["systems"])]
    counts = [int(round(c)) for c in np.exp(rng.uniform(np.log(64), np.log(2048), size=case["systems"]))]
    kT = [float(t) for t in rng.uniform(0.5, 2.0, size=case["systems"])]
    return edges, counts, kT


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "cycles": case.get("cycles", 0)}
    if kind in ("chain", "step", "mobility", "stokes"):
        s["own"] = _mg(case, seed)
        s["h"] = s["own"].h
        s["X"] = _particles(case["particles"], case["dim"], case["n"], seed)
        s["F"] = _forces(case["particles"], case["dim"], seed)
        s["U"] = torch.empty_like(s["X"])
        s["dt"] = 0.02 / case["n"] ** 2
        if kind == "chain":
            s["xi"] = torch.empty(s["own"].layout()[1], dtype=torch.float64, device="cuda")
    elif kind == "vcycle":
        s["own"] = _mg(case, seed)
        s["h"] = s["own"].h
        size, dtype = s["own"].layout()[1], s["own"].inner_dtype()
        s["v"], s["b"], s["cycle"] = _field(size, seed, dtype), _field(size, seed + 7919, dtype), 0
    elif kind in ("comp_sample", "comp_solve"):
        s["own"] = _comp(case, seed)
        s["h"] = s["own"].h
        size = S.selm_comp_size(s["h"])
        s["z"] = torch.zeros(size, dtype=torch.float64, device="cuda")
        if kind == "comp_solve":
            s["b"] = _field(size, seed, torch.float64)
    elif kind in ("mac_step", "mac_sample"):
        s["own"] = _mac(case, seed)
        s["h"] = s["own"].h
        if kind == "mac_step":
            s["X"] = _particles(case["particles"], case["dim"], 2 * case["n"], seed)
            s["F"] = _forces(case["particles"], case["dim"], seed)
            s["dt"] = 0.02 / (2 * case["n"]) ** 2
        else:
            s["xi"] = torch.empty(S.selm_mac_faces(s["h"]), dtype=torch.float64, device="cuda")
    elif kind == "batch":
        edges, counts, kT = _mix(case)
        descs = [S.make_desc(dim=3, n=e, kT=t, precision=S.SELM_FP32_REFINE64, seed=seed + i, instance=i,
                             max_particles=2048) for i, (e, t) in enumerate(zip(edges, kT))]
        s["own"] = _Owner(S.selm_batch_create(descs), S.selm_batch_destroy)
        s["h"] = s["own"].h
        S.selm_batch_autotune(s["h"])   # what a program that steps a batch many times does once
        s["X"] = [_particles(c, 3, e, seed + i) for i, (c, e) in enumerate(zip(counts, edges))]
        s["F"] = [_forces(c, 3, seed + i) for i, c in enumerate(counts)]
        s["dt"] = 0.02 / 128 ** 2
    else:
        raise ValueError(kind)
    return s


def run(state):
    s, kind = state, state["kind"]
    if kind == "chain":
        S.selm_mg_sample(s["h"], s["X"], s["cycles"], s["U"], xi_out=s["xi"])
        return {"g": s["U"], "xi": s["xi"]}
    if kind == "vcycle":
        S.selm_mg_vcycle(s["h"], S.SELM_SYS_VELOCITY, s["v"], s["b"], s["cycle"], 1)
        s["cycle"] += 1   # the next pass of the chain draws its own noise
        return {"v": s["v"]}
    if kind == "step":
        S.selm_mg_step(s["h"], s["X"], s["F"], s["dt"], 1, s["cycles"])
        return {"X": s["X"]}
    if kind == "mobility":
        S.selm_mg_solve(s["h"], s["X"], s["F"], s["U"], want_stats=False)
        return {"U": s["U"]}
    if kind == "stokes":
        S.selm_mg_stokes_mobility(s["h"], s["X"], s["F"], s["U"])
        return {"U": s["U"]}
    if kind == "comp_sample":
        S.selm_comp_sample(s["h"], s["cycles"], xi_out=s["z"])
        return {"xi": s["z"]}
    if kind == "comp_solve":
        s["z"].zero_()
        S.selm_comp_solve(s["h"], s["z"], s["b"], 1e-10, 100)
        return {"z": s["z"]}
    if kind == "mac_step":
        S.selm_mac_step(s["h"], s["X"], s["F"], s["dt"], 1, s["cycles"])
        return {"X": s["X"]}
    if kind == "mac_sample":
        S.selm_mac_sample(s["h"], s["cycles"], xi_out=s["xi"])
        return {"xi": s["xi"]}
    S.selm_batch_step(s["h"], s["X"], s["F"], s["dt"], 1, s["cycles"])
    return {"X": s["X"]}


# -- what a pass cannot do without ---------------------------------------------------------------------------
def _uniform(dim, n):
    return dim * n ** dim - n ** (dim - 1)   # the wall-normal component has one row less


def work(case):
    """Bytes: each persistent field that the pass advances read and written once, each other input and output
    once.  Operations: the 7-point row (5-point in 2-D) of every unknown in four sweeps, one residual in the
    V-cycle and one outside it, for the cycles asked for or for the seven a solve to 1e-10 takes, with the
    coarser levels' geometric sum."""
    kind, dim = case["kind"], case.get("dim", 3)
    if kind == "batch":
        edges, counts, _ = _mix(case)
        unknowns, particles = sum(_uniform(3, e) for e in edges), 3 * sum(counts)
    elif kind in ("comp_sample", "comp_solve"):
        n, K = case["n"], case["K"]
        unknowns = case["ncomp"] * n ** (dim - 1) * ((n - 1 - K) + K * 2 ** dim)
        particles = 0
    elif kind in ("mac_step", "mac_sample"):
        n, K = case["n"], case["K"]
        unknowns = dim * n ** (dim - 1) * ((n - K) + K * 2 ** dim)
        particles = dim * case.get("particles", 0)
    else:
        unknowns, particles = _uniform(dim, case["n"]), dim * case.get("particles", 0)
    solve = 0 if kind in ("chain", "vcycle", "comp_sample", "mac_sample") else 7
    cycles = solve + (1 if kind == "vcycle" else case.get("cycles", 0))
    row = 2 * (2 * dim + 1)
    flops = cycles * unknowns * row * 6 * 2 ** dim / (2 ** dim - 1)
    each = 4 if case.get("precision", "fp32") == "fp32" else 8
    if kind == "vcycle":
        size = 3 * each * unknowns                   # v in and out, b
    elif kind == "comp_solve":
        size = 16 * unknowns                         # b in, z out
    elif kind in ("chain", "comp_sample", "mac_sample"):
        size = 24 * unknowns                         # the chain read and written, its copy
    elif kind in ("mobility", "stokes"):
        size = 16 * unknowns                         # the force and the velocity field
    else:
        size = 32 * unknowns                         # these and the chain read and written
    return {"bytes": size + 8 * 3 * particles, "flops": flops}


# -- the channel's linear operators in 64 bits, by their eigenvectors ----------------------------------------
# Periodic axes by FFT, the wall axis by its sine or cosine vectors; s = mu h^(d-2) scales the Laplacian.
_CELL, _NODE, _NEUMANN = 0, 1, 2   # wall axis: cell centres (no slip), faces between cells, cell centres (no flux)


def _wall_vectors(kind, n, device):
    j = torch.arange(n, dtype=torch.float64, device=device)
    if kind == _CELL:
        m, x, f = j + 1, j + 0.5, torch.sin
    elif kind == _NODE:
        m, x, f = j[1:], j[1:], torch.sin
    else:
        m, x, f = j, j + 0.5, torch.cos
    Q = f(math.pi / n * x[:, None] * m[None, :])
    return Q / Q.norm(dim=0, keepdim=True), 2 - 2 * torch.cos(math.pi / n * m)


def _inverse(b, kind, n, dim, s):
    """The operator's (pseudo-)inverse on one component [nz, ny, nx]."""
    Q, lz = _wall_vectors(kind, n, b.device)
    lx = 2 - 2 * torch.cos(2 * math.pi / n * torch.arange(n, dtype=torch.float64, device=b.device))
    ly = lx if dim == 3 else torch.zeros(1, dtype=torch.float64, device=b.device)
    lam = s * (lz[:, None, None] + ly[None, :, None] + lx[None, None, :])
    t = torch.einsum("zm,zyx->myx", Q, b)
    t = torch.fft.fft2(t)
    t = t / torch.where(lam > 1e-14 * s, lam, torch.full_like(lam, math.inf))
    return torch.einsum("zm,myx->zyx", Q, torch.fft.ifft2(t).real)


def _kinds(dim):
    return [_CELL] * (dim - 1) + [_NODE]


def _solve_velocity(w, n, dim):
    s = float(n) ** (2 - dim)
    return [_inverse(c, k, n, dim, s) for c, k in zip(w, _kinds(dim))]


def _div(w, dim):
    out = torch.roll(w[0], -1, 2) - w[0]
    if dim == 3:
        out = out + torch.roll(w[1], -1, 1) - w[1]
    out[:-1] += w[-1]
    out[1:] -= w[-1]
    return out


def _div_t(p, dim):
    g = [torch.roll(p, 1, 2) - p]
    if dim == 3:
        g.append(torch.roll(p, 1, 1) - p)
    return g + [p[:-1] - p[1:]]


def _project(w, n, dim):
    phi = _inverse(_div(w, dim), _NEUMANN, n, dim, 1.0)
    return [a - b for a, b in zip(w, _div_t(phi, dim))]


def _stokes(f, n, dim):
    """A u + D^T p = f, D u = 0: conjugate gradients on D A^-1 D^T, whose condition is a small constant."""
    p = torch.zeros_like(_div(f, dim))
    r = _div(_solve_velocity(f, n, dim), dim)
    d, rr = r.clone(), (r * r).sum()
    stop = 1e-28 * rr
    for _ in range(200):
        if rr <= stop:
            break
        q = _div(_solve_velocity(_div_t(d, dim), n, dim), dim)
        a = rr / (d * q).sum()
        p, r = p + a * d, r - a * q
        r = r - r.mean()
        rr, old = (r * r).sum(), rr
        d = r + rr / old * d
    return _solve_velocity([a - b for a, b in zip(f, _div_t(p, dim))], n, dim)


def _peskin(r):
    r = r.abs()
    near = (3 - 2 * r + torch.sqrt((1 + 4 * r - 4 * r * r).clamp_min(0))) / 8
    far = (5 - 2 * r - torch.sqrt((-7 + 12 * r - 4 * r * r).clamp_min(0))) / 8
    return torch.where(r <= 1, near, torch.where(r <= 2, far, torch.zeros_like(r)))


def _nodes(X, c, n, dim):
    """Flat node numbers and weights [np, 4^dim] of velocity component c."""
    flat = torch.zeros((X.shape[0], 1), dtype=torch.int64, device=X.device)
    weight = torch.ones((X.shape[0], 1), dtype=torch.float64, device=X.device)
    for a in range(dim - 1, -1, -1):   # wall axis first: it is the slowest
        off = 0.0 if a == c else 0.5
        x = X[:, a] * n - off
        m = (torch.floor(x).to(torch.int64) - 1)[:, None] + torch.arange(4, device=X.device)
        w = _peskin(x[:, None] - m)
        if a < dim - 1:
            i, size = m % n, n
        else:
            lo, hi = (1, n - 1) if c == a else (0, n - 1)
            w = torch.where((m >= lo) & (m <= hi), w, torch.zeros_like(w))
            i, size = m.clamp(lo, hi) - lo, hi - lo + 1
        flat = (flat[:, :, None] * size + i[:, None, :]).reshape(X.shape[0], -1)
        weight = (weight[:, :, None] * w[:, None, :]).reshape(X.shape[0], -1)
    return flat, weight


def exact(case, seed):
    """The linear operations of the uniform channel.  A stochastic cycle has no value apart from its own noise and
    hierarchy, and the composite grids' operators have no eigenvectors in closed form: None."""
    if case["kind"] not in ("mobility", "stokes"):
        return None
    n, dim = case["n"], case["dim"]
    X, F = _particles(case["particles"], dim, n, seed), _forces(case["particles"], dim, seed)
    nodes = [_nodes(X, c, n, dim) for c in range(dim)]
    w = []
    for c, (flat, weight) in enumerate(nodes):
        shape = (n - 1 if c == dim - 1 else n, n if dim == 3 else 1, n)
        b = torch.zeros(math.prod(shape), dtype=torch.float64, device=X.device)
        b.index_add_(0, flat.reshape(-1), (weight * F[:, c:c + 1]).reshape(-1))
        w.append(b.reshape(shape))
    if case["kind"] == "stokes":
        u = _stokes(w, n, dim)
    else:
        if case["projection"]:
            w = _project(w, n, dim)
        u = _solve_velocity(w, n, dim)
        if case["projection"]:
            u = _project(u, n, dim)
    return {"U": torch.stack([(f.reshape(-1)[flat] * weight).sum(1) for f, (flat, weight) in zip(u, nodes)], dim=1)}
