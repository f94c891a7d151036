"""The work that is measured: exchange builds, their gradients and the calls around them.

A case is one synthetic solid (the fcc two-atom cell of the workloads package: seeded
orthonormal orbitals over ladders of Gaussian shells) and the call that a program makes on it:

    build     Plan.build: K_{mu i}, K and E_x, the call of every SCF iteration
    grad      exchange_build + backward: the gradients of a loss of K and E_x
    egrad     exchange_energy + backward: dE_x/dC (and dE_x/domega)
    orbitals  Plan.orbitals: the occupied orbitals on the grid
    bands     exchange of chosen conduction bands, then the paper-form assembly
    batch     several uneven cells in one launch

Sizes are those of the repository's configurations (cfg1 .. cfg5, a Gamma cell to the 350-AO
bench cell) and what lies between them. Plans are kept, as a program that iterates keeps them;
the coefficients C come from the seed. ``exact`` restates the method in plain 64-bit torch.
"""
import functools
import math

import numpy as np
import torch

import paper_2207_09028_gb300 as occri
from workloads import (analytic_overlap, fcc_cell, gamma_mesh, lowdin_orthonormalize,
                       make_shells, random_coefficients)

EDGES = (8, 9, 10, 12, 15, 16, 18, 20, 24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64)

# The five cells of a lattice-constant scan: edge (A), mesh, shells per l, nocc, grid.
SCAN = ((3.57, (3, 3, 3), (6, 5, 1), 4, 30), (4.05, (3, 3, 2), (9, 5, 3), 4, 32),
        (5.43, (2, 2, 2), (9, 6, 5), 4, 36), (5.65, (2, 2, 2), (11, 8, 6), 8, 40),
        (6.48, (2, 2, 2), (11, 8, 8), 8, 45))


def _case(name, op, precision, a, mesh, shells, nocc, grid, kernel="coulomb", omega=0.0,
          g0_mode=0, lo=0.08, hi=30.0, bands=0, cells=0):
    case = {"op": op, "precision": precision, "a": a, "k1": mesh[0], "k2": mesh[1],
            "k3": mesh[2], "s": shells[0], "p": shells[1], "d": shells[2], "f": shells[3],
            "nocc": nocc, "grid": grid, "kernel": kernel, "omega": omega, "g0_mode": g0_mode,
            "lo": lo, "hi": hi, "bands": bands, "cells": cells}
    return dict(case, name=name) if name else case


def listed():
    return [
        # the smallest call: a Gamma-point cell (cfg1), all latency and launches
        _case("gamma_24_mixed", "build", "mixed", 5.43, (1, 1, 1), (7, 2, 0, 0), 4, 24,
              lo=0.1, hi=20.0),
        # the ordinary SCF iteration: 8 k-points, 104 AOs (cfg2), in the fast precision ...
        _case("k222_36_tc", "build", "mixed_tc", 5.43, (2, 2, 2), (9, 6, 5, 0), 4, 36),
        # ... and in double precision, the form others are checked with
        _case("k222_36_fp64", "build", "fp64", 5.43, (2, 2, 2), (9, 6, 5, 0), 4, 36),
        # a range-separated build on 64 k-points, 200 AOs (cfg3)
        _case("k444_48_erfc_tc", "build", "mixed_tc", 5.43, (4, 4, 4), (15, 10, 11, 0), 4, 48,
              "erfc", 0.11, 1),
        # the largest: the bench cell (350 AOs, nocc 8, 60^3) on 64 k-points
        _case("k444_60_tc", "build", "mixed_tc", 5.43, (4, 4, 4), (20, 14, 10, 9), 8, 60,
              lo=0.06, hi=40.0),
        # an odd grid edge and nocc 8 (the widest cell of cfg4), CUDA-core contraction
        _case("k222_45_erfc_mixed", "build", "mixed", 6.48, (2, 2, 2), (11, 8, 8, 0), 8, 45,
              "erfc", 0.11, 1),
        # an uneven mesh with the truncated Coulomb kernel and an odd nocc
        _case("k123_50_trunc_tc", "build", "mixed_tc", 5.43, (1, 2, 3), (9, 6, 5, 0), 5, 50,
              "coulomb_trunc", 0.0, 1),
        # a training step through K and E_x with a learned omega (the tightest cell of cfg4)
        _case("k333_30_grad_mixed", "grad", "mixed", 3.57, (3, 3, 3), (6, 5, 1, 0), 4, 30,
              "erfc", 0.11, 1),
        # fitting omega in double precision (the second cell of cfg4)
        _case("k332_32_egrad_fp64", "egrad", "fp64", 4.05, (3, 3, 2), (9, 5, 3, 0), 4, 32,
              "erfc", 0.11, 1),
        # orbitals for plotting or another code: the bench cell's basis on 8 k-points
        _case("k222_60_orbitals", "orbitals", "mixed", 5.43, (2, 2, 2), (20, 14, 10, 9), 8, 60,
              lo=0.06, hi=40.0),
        # a band structure: 4 occupied orbitals and 8 conduction bands (nocc 12 in the pair loop)
        _case("k222_40_bands_mixed", "bands", "mixed", 5.65, (2, 2, 2), (11, 8, 6, 0), 4, 40,
              bands=8),
        # a lattice-constant scan: the five cells of cfg4 in one launch
        _case("scan_batch_mixed", "batch", "mixed", 5.43, (2, 2, 2), (9, 6, 5, 0), 4, 36,
              "erfc", 0.11, 1, cells=5),
    ]


def _log_choice(rng, values):
    """One of the sorted values, even in the logarithm."""
    x = math.exp(rng.uniform(math.log(values[0]), math.log(values[-1])))
    return min(values, key=lambda v: abs(math.log(v / x)))


def draw(rng):
    while True:
        op = rng.choice(("build",) * 6 + ("grad", "egrad", "orbitals", "bands", "batch"))
        precision = rng.choice(("mixed", "mixed", "mixed_tc", "mixed_tc", "mixed_tc", "fp64"))
        mesh = tuple(rng.choice((1, 2, 2, 3, 4)) for _ in range(3))
        grid = _log_choice(rng, EDGES[4:])
        nocc = _log_choice(rng, tuple(range(1, 17)))
        kernel, omega, g0 = rng.choice((("coulomb", 0.0, 0), ("coulomb", 0.0, 0),
                                        ("erfc", round(rng.uniform(0.1, 0.4), 3), 1),
                                        ("erf", round(rng.uniform(0.1, 0.4), 3), 0),
                                        ("coulomb_trunc", 0.0, 1)))
        shells = (rng.randint(6, 20), rng.randint(2, 14), rng.choice((0, rng.randint(1, 11))),
                  rng.choice((0, 0, rng.randint(1, 9))))
        case = _case(None, op, precision, round(rng.uniform(3.6, 6.5), 2), mesh, shells, nocc,
                     grid, kernel, omega, g0, lo=0.08, hi=30.0,
                     bands=rng.randint(1, 8) if op == "bands" else 0,
                     cells=rng.randint(2, 4) if op == "batch" else 0)
        if op == "batch" and precision == "fp64":
            continue
        if 2e5 < _cost(case) < 8e9 and _nao(case) >= 2 * (nocc + case["bands"]):
            return case


# ---------------------------------------------------------------- the problem of a case

def _cells(case):
    """The cells of a case: one, or for a batch those of the scan, or `cells` like the case's own
    with other edges and grids."""
    if not case["cells"]:
        return [dict(case)]
    if case["cells"] == 5:
        return [dict(case, a=a, k1=m[0], k2=m[1], k3=m[2], s=n[0], p=n[1], d=n[2], f=0,
                     nocc=no, grid=g) for a, m, n, no, g in SCAN]
    near = EDGES.index(case["grid"])
    return [dict(case, a=round(case["a"] + 0.2 * i, 2), grid=EDGES[max(0, near - i)])
            for i in range(case["cells"])]


def _nao(c):
    return 2 * (c["s"] + 3 * c["p"] + 5 * c["d"] + 7 * c["f"])


def _nk(c):
    return c["k1"] * c["k2"] * c["k3"]


def _fields(c, nocc):
    """Pair densities of one build: (k, k', i, j), each with its conjugate counted once."""
    n = _nk(c) * nocc
    return n * (n + 1) // 2


def _cost(case):
    """Points of pair fields in one pass, weighted by precision: what draw() bounds."""
    total = 0.0
    for c in _cells(case):
        n = c["nocc"] + c["bands"]
        rounds = {"build": 1, "batch": 1, "orbitals": 0.01, "egrad": 2, "grad": 4,
                  "bands": 2}[case["op"]]
        total += rounds * _fields(c, n) * c["grid"] ** 3 * (60 if c["precision"] == "fp64" else 1)
    return total


@functools.lru_cache(maxsize=32)
def _geometry(a, mesh, shells, lo, hi):
    lattice, xyz = fcc_cell(a)
    sa, sl, sx = make_shells(2, shells, lo, hi)
    kfrac = gamma_mesh(*mesh)
    return lattice, xyz, sa, sl, sx, kfrac, analytic_overlap(lattice, xyz, sa, sl, sx, kfrac)


def _geometry_of(c):
    return _geometry(c["a"], (c["k1"], c["k2"], c["k3"]), (c["s"], c["p"], c["d"], c["f"]),
                     c["lo"], c["hi"])


def _inputs(case, seed):
    """Per cell: orthonormal C [nk, nao, nocc + bands] (real at Gamma alone), and for a gradient
    the Hermitian weights of K in the loss."""
    out = []
    for n, c in enumerate(_cells(case)):
        s = _geometry_of(c)[6]
        rng = np.random.default_rng([seed, n])
        C = lowdin_orthonormalize(random_coefficients(rng, _nk(c), _nao(c),
                                                      c["nocc"] + c["bands"], _nk(c) > 1), s)
        w = None
        if case["op"] == "grad":
            w = random_coefficients(rng, _nk(c), _nao(c), _nao(c), _nk(c) > 1) / _nao(c)
            w = w + np.conj(np.swapaxes(w, 1, 2))
        out.append((C, w))
    return out


def _plan(c, nocc):
    lattice, xyz, sa, sl, sx, kfrac, _ = _geometry_of(c)
    return occri.Plan(lattice, xyz, sa, sl, sx, kfrac, nocc, (c["grid"],) * 3, c["kernel"],
                      c["omega"], c["g0_mode"], c["precision"])


# ---------------------------------------------------------------- prepare and run

def prepare(case, seed):
    dev = torch.device("cuda")
    cells = _cells(case)
    given = [(torch.from_numpy(C).to(dev), None if w is None else torch.from_numpy(w).to(dev))
             for C, w in _inputs(case, seed)]
    state = {"op": case["op"], "C": [C for C, _ in given], "w": given[0][1]}
    if case["op"] == "bands":
        c = cells[0]
        state["plans"] = [_plan(c, c["nocc"]), _plan(c, c["nocc"] + c["bands"]),
                          _plan(c, c["bands"])]
        state["occ"] = state["C"][0][:, :, :c["nocc"]].contiguous()
        state["S"] = torch.from_numpy(_geometry_of(c)[6]).to(dev).contiguous()
        return state
    state["plans"] = [_plan(c, c["nocc"]) for c in cells]
    if case["op"] == "batch":
        state["batch"] = occri.Batch(state["plans"])
        z = [dict(dtype=torch.complex128, device=dev) for _ in cells]
        state["KC"] = [torch.empty_like(C) for C in state["C"]]
        state["K"] = [torch.empty((C.shape[0], C.shape[1], C.shape[1]), **o)
                      for C, o in zip(state["C"], z)]
        state["Ex"] = [torch.zeros(1, dtype=torch.float64, device=dev) for _ in cells]
    if case["op"] in ("grad", "egrad"):
        state["C"][0].requires_grad_(True)
        state["omega"] = None
        if case["kernel"] in ("erfc", "erf"):
            state["omega"] = torch.tensor(case["omega"], dtype=torch.float64, device=dev,
                                          requires_grad=True)
    return state


def run(state):
    op, plan, C = state["op"], state["plans"][0], state["C"][0]
    if op == "build":
        KC, K, Ex = plan.build(C)
        return {"KC": KC, "K": K, "Ex": Ex}
    if op == "orbitals":
        return {"psi": plan.orbitals(C)}
    if op == "batch":
        state["batch"].build(state["C"], state["KC"], state["K"], state["Ex"])
        return {"KC": state["KC"], "K": state["K"], "Ex": state["Ex"]}
    if op == "bands":
        KC, _, Ex = plan.build(state["occ"], want_k=False)
        KCr = state["plans"][1].k_build_conduction(state["plans"][2], C)
        K = plan.assemble_paper(state["S"], C, torch.cat((KC, KCr), dim=2))
        return {"KC": KC, "KCr": KCr, "K": K, "Ex": Ex}
    C.grad = None
    w = state["omega"]
    if w is not None:
        w.grad = None
    if op == "grad":
        K, Ex = occri.exchange_build(plan, C, w)
        (Ex + 0.1 * (state["w"].conj() * K).real.sum()).backward()
        out = {"K": K.detach(), "Ex": Ex.detach(), "gC": C.grad}
    else:
        Ex = occri.exchange_energy(plan, C, w)
        Ex.backward()
        out = {"Ex": Ex.detach(), "gC": C.grad}
    if w is not None:
        out["gomega"] = w.grad
    return out


def work(case):
    """Flops: two FFTs (5 N log2 N each), the density, the kernel and the accumulations per pair
    field, and the two products with the AOs. Bytes: C in, the results out."""
    flops = nbytes = 0.0
    for c in _cells(case):
        nk, nao, ng = _nk(c), _nao(c), c["grid"] ** 3
        per_field = 10 * ng * math.log2(ng) + (6 + 2 + 16) * ng
        aos = 8.0 * nk * nao * ng   # one product of the AOs with one orbital
        n = c["nocc"] + c["bands"]
        op = case["op"]
        if op == "orbitals":
            flops += aos * n
            nbytes += 16.0 * nk * n * (nao + ng)
            continue
        flops += _fields(c, c["nocc"]) * per_field + 2 * aos * c["nocc"]
        nbytes += 16.0 * nk * nao * (n + c["nocc"] + (nao if op != "egrad" else 0)) + 8
        if op == "bands":   # the bands' columns: densities of occupied orbitals with bands
            flops += (nk * nk * c["nocc"] * c["bands"] * per_field +
                      2 * aos * c["bands"] + 16.0 * nk * nao * nao * n)
            nbytes += 16.0 * nk * nao * (nao + c["bands"])
        if op == "grad":    # two round trips per pair, orbitals of the adjoint, contraction
            flops += 2 * _fields(c, c["nocc"]) * per_field + 3 * aos * c["nocc"]
            nbytes += 16.0 * nk * nao * (nao + c["nocc"])
        if op == "egrad" and c["kernel"] in ("erfc", "erf"):
            flops += _fields(c, c["nocc"]) * (5 * ng * math.log2(ng) + 10 * ng)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # Against exact(): 2e-7 to 7e-7 in the mixed precisions (largest in the bands' columns, a
    # difference of two builds, and in K, which adds the condition of C^H K C), up to 1e-14 in
    # FP64 on the listed cases; the drawn ones reach worse conditions of C^H K C.
    return {"rel": 1e-12, "max": 1e-10} if case["precision"] == "fp64" else {"rel": 4e-6,
                                                                             "max": 2e-4}


# ---------------------------------------------------------------- the method in 64 bits

_POLY = {   # real solid harmonics, m = -l .. l
    0: [lambda x, y, z: torch.ones_like(x)],
    1: [lambda x, y, z: x, lambda x, y, z: y, lambda x, y, z: z],
    2: [lambda x, y, z: x * y, lambda x, y, z: y * z,
        lambda x, y, z: 2 * z * z - x * x - y * y, lambda x, y, z: x * z,
        lambda x, y, z: x * x - y * y],
    3: [lambda x, y, z: y * (3 * x * x - y * y), lambda x, y, z: x * y * z,
        lambda x, y, z: y * (4 * z * z - x * x - y * y),
        lambda x, y, z: z * (2 * z * z - 3 * x * x - 3 * y * y),
        lambda x, y, z: x * (4 * z * z - x * x - y * y), lambda x, y, z: z * (x * x - y * y),
        lambda x, y, z: x * (x * x - 3 * y * y)],
}
# integral of P_lm(u)^2 over the unit sphere; a primitive's norm follows from the radial integral
_SPHERE = {0: [4 * math.pi], 1: [4 * math.pi / 3] * 3,
           2: [4 * math.pi / 15] * 2 + [16 * math.pi / 5] + [4 * math.pi / 15, 16 * math.pi / 15],
           3: [32 * math.pi / 35, 4 * math.pi / 105, 32 * math.pi / 21, 16 * math.pi / 7,
               32 * math.pi / 21, 16 * math.pi / 105, 32 * math.pi / 35]}


def _norm(l, m, alpha):
    radial = math.gamma(l + 1.5) / (2.0 * (2.0 * alpha) ** (l + 1.5))
    return 1.0 / math.sqrt(_SPHERE[l][m] * radial)


def _grid_points(c, dev):
    n = torch.arange(c["grid"], dtype=torch.float64, device=dev) / c["grid"]
    f = torch.stack(torch.meshgrid(n, n, n, indexing="ij"), -1).reshape(-1, 3)
    return f, f @ torch.from_numpy(_geometry_of(c)[0]).to(dev)


def _bloch_aos(c, dev):
    """chi [nk, nao, ng]: sum over lattice vectors T of e^{ik.T} phi(r - A - T)."""
    lattice, xyz, sa, sl, sx, kfrac, _ = _geometry_of(c)
    _, r = _grid_points(c, dev)
    ng = r.shape[0]
    chi = torch.zeros((len(kfrac), _nao(c), ng), dtype=torch.complex128, device=dev)
    reach = float(np.linalg.norm(lattice.sum(0)))
    centre = 0.5 * lattice.sum(0)
    ao = 0
    for a, l, alpha in zip(sa, sl, sx):
        l, alpha = int(l), float(alpha)
        rc = math.sqrt(46.0 / alpha) + l
        span = int(math.ceil((rc + reach) * np.linalg.norm(np.linalg.inv(lattice), axis=0).max())) + 2
        n = np.arange(-span, span + 1)
        n = np.stack(np.meshgrid(n, n, n, indexing="ij"), -1).reshape(-1, 3)
        T = n @ lattice
        keep = np.linalg.norm(T + xyz[a] - centre, axis=1) <= rc + 0.51 * reach
        n, T = n[keep], torch.from_numpy(T[keep]).to(dev)
        ph = np.exp(2j * np.pi * (kfrac @ n.T))
        ph = torch.from_numpy(np.concatenate((ph.real, ph.imag))).to(dev)    # [2 nk, nT]
        acc = torch.zeros((2 * len(kfrac), (2 * l + 1) * ng), dtype=torch.float64, device=dev)
        step = max(1, int(2.5e8 // ((2 * l + 1) * ng)))
        for t in range(0, len(T), step):
            d = r[None] - torch.from_numpy(xyz[a]).to(dev) - T[t:t + step, None]
            x, y, z = d[..., 0], d[..., 1], d[..., 2]
            e = torch.exp(-alpha * (x * x + y * y + z * z))
            phi = torch.stack([_norm(l, m, alpha) * P(x, y, z) * e
                               for m, P in enumerate(_POLY[l])], 1)
            acc += ph[:, t:t + step] @ phi.reshape(phi.shape[0], -1)
        acc = acc.reshape(2, len(kfrac), 2 * l + 1, ng)
        chi[:, ao:ao + 2 * l + 1] = torch.complex(acc[0], acc[1])
        ao += 2 * l + 1
    return chi


def _kernel(c, q, omega, dev):
    """v(|G+q|) on the FFT bins [N, N, N]; tied aliases averaged, g0 at G+q = 0."""
    lattice = _geometry_of(c)[0]
    B = torch.from_numpy(2 * np.pi * np.linalg.inv(lattice).T).to(dev)
    N, D = c["grid"], (c["k1"], c["k2"], c["k3"])
    volume = abs(np.linalg.det(lattice)) * D[0] * D[1] * D[2]
    rc = (3 * volume / (4 * math.pi)) ** (1.0 / 3.0)
    axes, tied = [], []
    for d in range(3):   # integers X = (m + q) D, reduced to [-N D / 2, N D / 2)
        P = N * D[d]
        X = np.arange(N) * D[d] + int(round(q[d] * D[d]))
        X = (2 * X + P) // (2 * P) * -P + X
        axes.append((X, np.where(2 * X == -P, X + P, X)))
        tied.append(2 * X == -P)
    v = torch.zeros((N, N, N), dtype=torch.float64, device=dev)
    for alias in range(8):
        ax = [torch.from_numpy(axes[d][(alias >> d) & 1] / D[d]).to(dev) for d in range(3)]
        x = torch.stack(torch.meshgrid(*ax, indexing="ij"), -1) @ B
        g2 = (x * x).sum(-1)
        zero = g2 < 1e-14
        g = torch.where(zero, torch.ones_like(g2), g2)
        kind = c["kernel"]
        if kind == "coulomb":
            f, f0 = 4 * math.pi / g, 0.0
        elif kind == "coulomb_trunc":
            f, f0 = 4 * math.pi / g * (1 - torch.cos(torch.sqrt(g) * rc)), 2 * math.pi * rc * rc
        elif kind == "erfc":
            f, f0 = -4 * math.pi / g * torch.expm1(-g / (4 * omega * omega)), math.pi / omega ** 2
        else:
            f, f0 = 4 * math.pi / g * torch.exp(-g / (4 * omega * omega)), 0.0
        v = v + torch.where(zero, f0 if c["g0_mode"] else 0.0, f) / 8
    return v


def _columns(c, chi, C, density, omega):
    """K_{mu i}(k) of the orbitals C with the exchange of the orbitals `density`."""
    kfrac = _geometry_of(c)[5]
    dev, N, nk = C.device, c["grid"], len(kfrac)
    f, _ = _grid_points(c, dev)
    ph = torch.exp(2j * math.pi * (torch.from_numpy(kfrac).to(dev) @ f.T))   # e^{ik.r}

    def periodic(X):
        return torch.stack([(X[k].T @ chi[k]) * ph[k].conj() for k in range(nk)])

    u = periodic(C)
    d = u if density is C else periodic(density)
    table = {}

    def kernel(k, p):
        q = tuple(kfrac[k] - kfrac[p])
        if omega is not None and torch.is_tensor(omega) and omega.requires_grad:
            return _kernel(c, q, omega, dev)
        key = tuple(np.round(q, 9))
        if key not in table:
            table[key] = _kernel(c, q, omega, dev)
        return table[key]

    def one(k, u, d, omega):
        y = 0
        for p in range(nk):
            rho = d[p].conj()[None] * u[k][:, None]
            g = torch.fft.fftn(rho.reshape(*rho.shape[:2], N, N, N), dim=(2, 3, 4))
            w = torch.fft.ifftn(g * kernel(k, p), dim=(2, 3, 4)).reshape(rho.shape)
            y = y + (w * d[p][None]).sum(1)
        return chi[k].conj() @ (y * ph[k]).T

    scale = -abs(np.linalg.det(_geometry_of(c)[0])) / (nk * N ** 3)
    cols = []
    for k in range(nk):
        if torch.is_grad_enabled() and C.requires_grad:
            cols.append(torch.utils.checkpoint.checkpoint(one, k, u, d, omega,
                                                          use_reentrant=False))
        else:
            cols.append(one(k, u, d, omega))
    return scale * torch.stack(cols)


def _assembled(C, KC):
    M = C.conj().transpose(1, 2) @ KC
    M = 0.5 * (M + M.conj().transpose(1, 2))
    Ex = M.diagonal(dim1=1, dim2=2).real.sum() / C.shape[0]
    return KC @ torch.linalg.solve(M, KC.conj().transpose(1, 2)), Ex


def _exact_seconds(case):
    """About what exact() takes: 64-bit transforms over the ordered pairs and the AO sums."""
    total = 0.0
    for c in _cells(case):
        n, nk, ng = c["nocc"] + c["bands"], _nk(c), c["grid"] ** 3
        rounds = {"orbitals": 0, "grad": 5, "egrad": 5}.get(case["op"], 1)
        total += rounds * nk * nk * (n * n * ng * 1.2e-9 + 1e-3)
        total += 300.0 * _nao(c) * ng * (8 * nk + 400) / 1e12
    return total


def exact(case, seed):
    if _exact_seconds(case) > 14.0:
        return None
    import torch.utils.checkpoint  # noqa: F401
    dev = torch.device("cuda")
    op, results = case["op"], []
    for c, (C, w) in zip(_cells(case), _inputs(case, seed)):
        C = torch.from_numpy(C).to(dev)
        chi = _bloch_aos(c, dev)
        omega = c["omega"]
        if op == "orbitals":
            psi = torch.stack([C[k].T @ chi[k] for k in range(_nk(c))])
            return {"psi": psi.reshape(_nk(c), c["nocc"], *(c["grid"],) * 3)}
        if op in ("grad", "egrad"):
            C.requires_grad_(True)
            if c["kernel"] in ("erfc", "erf"):
                omega = torch.tensor(omega, dtype=torch.float64, device=dev, requires_grad=True)
            K, Ex = _assembled(C, _columns(c, chi, C, C, omega))
            loss = Ex
            if op == "grad":
                loss = Ex + 0.1 * (torch.from_numpy(w).to(dev).conj() * K).real.sum()
            loss.backward()
            out = {"K": K.detach(), "Ex": Ex.detach(), "gC": C.grad}
            if op == "egrad":
                del out["K"]
            if torch.is_tensor(omega):
                out["gomega"] = omega.grad
            return out
        with torch.no_grad():
            occ = C[:, :, :c["nocc"]].contiguous()
            KC = _columns(c, chi, occ, occ, omega)
            K, Ex = _assembled(occ, KC)
            if op == "bands":
                KCr = _columns(c, chi, C[:, :, c["nocc"]:].contiguous(), occ, omega)
                full = torch.cat((KC, KCr), dim=2)
                SC = torch.from_numpy(_geometry_of(c)[6]).to(dev) @ C
                M = C.conj().transpose(1, 2) @ full
                M = 0.5 * (M + M.conj().transpose(1, 2))
                h = SC.conj().transpose(1, 2)
                K = full @ h + SC @ full.conj().transpose(1, 2) - SC @ M @ h
                return {"KC": KC, "KCr": KCr, "K": K, "Ex": Ex.reshape(1)}
            results.append((KC, K, Ex.reshape(1)))
            del chi
    if op == "batch":
        return {n: [x[i] for x in results] for i, n in enumerate(("KC", "K", "Ex"))}
    return dict(zip(("KC", "K", "Ex"), results[0]))
