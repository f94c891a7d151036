"""Bloch AOs in tiles (csrc/occri_chi.cu) where they change form: the transform over classes at
one class, full and partly filled axes and columns that take a part of a shell; meshes it does
not take, with entries that run out; lists too long for shared memory, ragged point blocks,
every width of the products. Orbitals and K_{mu i} against the oracle."""
import dataclasses

import numpy as np
import pytest

import oracle as O
from workloads import small_workload
from workloads.synthetic import (analytic_overlap, lowdin_orthonormalize, random_coefficients)

pytestmark = pytest.mark.gpu

CASES = {
    # Gamma: one class, several CTAs per block
    "gamma": dict(mesh=(1, 1, 1), grid=(9, 9, 9), counts=(3, 2), lo=0.1, nocc=1),
    # even and odd axes of the transform, wide and narrow shells side by side
    "even": dict(mesh=(1, 4, 2), grid=(10, 10, 10), counts=(2, 2, 1), lo=0.1, nocc=5),
    "class8": dict(mesh=(2, 2, 2), grid=(9, 9, 9), counts=(2, 1, 1), lo=0.1, nocc=4),
    "odd": dict(mesh=(3, 3, 3), grid=(8, 8, 8), counts=(2, 1, 1, 1), lo=0.12, nocc=9),
    "wide": dict(mesh=(5, 1, 1), grid=(8, 8, 8), counts=(3, 2, 1), lo=0.2, nocc=17),
    # a length the transform does not take: an entry per image, more than fit
    "seven": dict(mesh=(1, 1, 7), grid=(8, 8, 8), counts=(2, 1, 1, 1), lo=0.12, nocc=3),
    # 100 classes: in FP64 an f shell does not fit the columns whole (orbitals only)
    "columns": dict(mesh=(5, 4, 5), grid=(8, 8, 8), counts=(2, 0, 0, 1), lo=0.12, nocc=2),
    # over 4,000 images in reach: the records stay in global memory
    "long_list": dict(mesh=(1, 1, 2), grid=(8, 8, 8), counts=(1, 1), a_ang=2.0, lo=0.05, hi=0.05,
                      nocc=1),
}


def _with_kfrac(w, kfrac):
    """The same cell at other k-points, with orthonormal orbitals there."""
    kfrac = np.asarray(kfrac, float)
    s = analytic_overlap(w.lattice, w.xyz, w.shell_atom, w.shell_l, w.shell_alpha, kfrac)
    x = random_coefficients(np.random.default_rng(3), len(kfrac), w.nao, w.nocc, True)
    return dataclasses.replace(w, kfrac=kfrac, C=lowdin_orthonormalize(x, s))


def _workload(name):
    if name == "off_mesh":   # two points of a 1/8 mesh: as many classes as images
        w = small_workload(mesh=(1, 1, 1), grid=(8, 8, 8), counts=(2, 1, 1), lo=0.15, nocc=2,
                           seed=31, complex_c=True)
        return _with_kfrac(w, [[0.125, 0.0, 0.375], [0.625, 0.25, 0.0]])
    w = small_workload(seed=31, **CASES[name])
    if name == "long_list":   # the AOs nearly cancel at k = 1/2: plain, not orthonormal, orbitals
        w = dataclasses.replace(w, C=np.full_like(w.C, 0.3 + 0.1j))
    return w


@pytest.mark.parametrize("name", list(CASES) + ["off_mesh"])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_orbitals_and_contraction_match_oracle(name, precision):
    import torch
    import paper_2207_09028_gb300 as occri
    w = _workload(name)
    chi = O.bloch_aos(w.lattice, w.xyz, w.shell_atom, w.shell_l, w.shell_alpha, w.kfrac,
                      grid=w.grid)
    psi = O.orbitals_on_grid(chi, w.C)
    plan = occri.Plan.from_workload(w, precision=precision)
    C = torch.from_numpy(w.C).cuda()
    got = plan.orbitals(C).cpu().numpy().reshape(psi.shape)
    # The rounding of a sequential sum of n images of one sign is at most n u of it, u = 1.1e-16
    # (FP64) or 6e-8 (FP32); the long list has n = 5,200 (FP64) or 4,000 (FP32) over two classes,
    # the other cells about 100. FP32 bars: n u = 2.4e-4 and 6e-6 at most; the random-walk sizes
    # sqrt(n) u = 4e-6 and 6e-7, with a margin of about 3, are asked for.
    bar = 1e-12 if precision == "fp64" else (1.2e-5 if name == "long_list" else 2e-6)
    assert np.abs(got - psi).max() <= bar * np.abs(psi).max()
    if name == "columns":
        return
    g0 = O.g0_value(w.kernel, w.omega, w.g0_mode, w.lattice, w.kfrac)
    kc = O.occri_kc(w.lattice, w.grid, w.kfrac, psi, chi, w.kernel, w.omega, g0)
    KC = plan.build(C)[0]
    # (The long list's orbital at Gamma is constant to 1e-4, so without its G = 0 term its density
    # is what the sums above round off: K is compared in FP64 there.)
    if name != "long_list" or precision == "fp64":
        tol = 1e-10 if precision == "fp64" else 1e-5   # four orbitals in each term
        assert np.abs(KC.cpu().numpy() - kc).max() <= tol * np.abs(kc).max()
    # the contraction adds its partial sums in a fixed order
    assert torch.equal(KC, plan.build(C)[0])


@pytest.fixture(scope="module")
def ragged():
    w = small_workload(mesh=(1, 2, 2), grid=(45, 45, 45), counts=(3, 1), lo=0.15, nocc=2, seed=37,
                       complex_c=True)
    return w, O.bloch_aos(w.lattice, w.xyz, w.shell_atom, w.shell_l, w.shell_alpha, w.kfrac,
                          grid=w.grid)


@pytest.mark.parametrize("nocc", [3, 7, 12])
def test_orbitals_two_blocks_per_warp(ragged, nocc):
    """Enough ragged blocks that a warp takes two (which differ in the AOs that reach them)."""
    import torch
    import paper_2207_09028_gb300 as occri
    w, chi = ragged
    c = np.random.default_rng(5).standard_normal((2, w.nk, w.nao, nocc))
    w = dataclasses.replace(w, nocc=nocc, C=c[0] + 1j * c[1])
    psi = O.orbitals_on_grid(chi, w.C)
    plan = occri.Plan.from_workload(w, precision="mixed")
    got = plan.orbitals(torch.from_numpy(w.C).cuda()).cpu().numpy().reshape(psi.shape)
    # the bar above: sqrt(n) u for n of about 100 images and AOs, with a margin of about 3
    assert np.abs(got - psi).max() <= 2e-6 * np.abs(psi).max()


def _half_shifted(n):
    ax = (np.arange(n) + 0.5) / n
    return np.stack(np.meshgrid(ax, ax, ax, indexing="ij"), -1).reshape(-1, 3)


MANY_K = {
    # a length that the transform does not take, k-points past a group of four; about 340 images,
    # four batches; groups of one to eight AOs (s and p together, d with s, f alone)
    "axis17": dict(kfrac=[[0, 0, j / 17] for j in range(17)], counts=(3, 2, 1, 1), lo=0.12),
    # several CTAs share the k-points
    "shifted": dict(kfrac=_half_shifted(4), counts=(2, 1, 1), lo=0.15),
    # one batch of a few images, blocks that some shells do not reach
    "tight": dict(kfrac=[[0, j / 16, 0.5] for j in range(16)], counts=(2, 2, 1), a_ang=6.0,
                  lo=0.4, hi=20.0),
}


@pytest.mark.parametrize("name", list(MANY_K))
def test_many_k_points_without_the_transform(name):
    """chi_dense_kernel (FP32) and a narrow shell's slices of the k-points (FP64) against the oracle,
    and the tiles in the contraction against FP64."""
    import torch
    import paper_2207_09028_gb300 as occri
    case = dict(MANY_K[name])
    kfrac = case.pop("kfrac")
    w = small_workload(mesh=(1, 1, 1), grid=(9, 9, 9), nocc=2, seed=33, complex_c=True, **case)
    w = _with_kfrac(w, kfrac)
    chi = O.bloch_aos(w.lattice, w.xyz, w.shell_atom, w.shell_l, w.shell_alpha, w.kfrac,
                      grid=w.grid)
    psi = O.orbitals_on_grid(chi, w.C)
    C = torch.from_numpy(w.C).cuda()
    # as above: sqrt(n) u with a margin of about 3, for n of about 350
    for precision, bar in (("fp64", 1e-12), ("mixed", 4e-6)):
        plan = occri.Plan.from_workload(w, precision=precision)
        got = plan.orbitals(C).cpu().numpy().reshape(psi.shape)
        assert np.abs(got - psi).max() <= bar * np.abs(psi).max(), precision
    ref = occri.Plan.from_workload(w, precision="fp64").build(C)[0]
    for precision in ("mixed", "mixed_tc"):
        kc = occri.Plan.from_workload(w, precision=precision).build(C)[0]
        assert (kc - ref).abs().max() <= 1e-5 * ref.abs().max()


@pytest.mark.parametrize("mesh", [(1, 1, 2), (1, 1, 3)])   # real and complex tiles
@pytest.mark.parametrize("precision", ["fp64", "mixed", "mixed_tc"])
def test_aos_in_chunks(precision, mesh):
    """Without the memory for all tiles a plan takes them in chunks: the same orbitals, and the same
    sums but for their order."""
    import torch
    import paper_2207_09028_gb300 as occri
    w = small_workload(mesh=mesh, grid=(15, 15, 15), counts=(3, 2, 1), nocc=3, seed=47)
    C = torch.from_numpy(w.C).cuda()
    rng = np.random.default_rng(8)
    G = torch.from_numpy(rng.standard_normal((w.nk, w.nao, w.nao)) + 0j).cuda()

    def results(plan):
        psi = plan.orbitals(C).clone()
        kc = plan.build(C)[0]
        return psi, kc, plan.vjp_full(C, 0.3, None, G), plan.info()["launches_per_build"]

    whole = results(occri.Plan.from_workload(w, precision=precision))
    for nth in range(1, 60):   # the first failure that a plan survives is that of its tiles
        occri.fail_allocation(nth)
        try:
            plan = occri.Plan.from_workload(w, precision=precision)
            break
        except occri.OccriError as e:
            assert e.status == occri.OCCRI_ENOMEM
        finally:
            occri.fail_allocation(0)
    parts = results(plan)
    assert parts[3] > whole[3]
    assert torch.equal(parts[0], whole[0])
    # FP32: sums of about 3,000 points in another order, sqrt(3000) u = 3.3e-6 at most
    tol = 1e-12 if precision == "fp64" else 3e-6
    for x, y in zip(parts[1:3], whole[1:3]):
        assert (x - y).abs().max() <= tol * y.abs().max()


@pytest.mark.parametrize("mesh,nocc", [((1, 1, 3), 12), ((1, 1, 3), 20), ((1, 1, 17), 9)])
def test_tensor_core_widths_on_complex_tiles(mesh, nocc):
    """The tensor-core contraction of 32 and 64 columns where the tiles are complex."""
    import torch
    import paper_2207_09028_gb300 as occri
    w = small_workload(mesh=mesh, grid=(9, 9, 9), counts=(6, 4, 1), nocc=nocc, seed=51)
    chi = O.bloch_aos(w.lattice, w.xyz, w.shell_atom, w.shell_l, w.shell_alpha, w.kfrac,
                      grid=w.grid)
    psi = O.orbitals_on_grid(chi, w.C)
    g0 = O.g0_value(w.kernel, w.omega, w.g0_mode, w.lattice, w.kfrac)
    kc = O.occri_kc(w.lattice, w.grid, w.kfrac, psi, chi, w.kernel, w.omega, g0)
    plan = occri.Plan.from_workload(w, precision="mixed_tc")
    assert plan.info()["contraction_tc"] == 1
    got = plan.build(torch.from_numpy(w.C).cuda())[0].cpu().numpy()
    # the bar of the other builds above: a few FP32 roundings of each of the four orbitals of a
    # term, at the size of the largest
    assert np.abs(got - kc).max() <= 1e-5 * np.abs(kc).max()


@pytest.mark.parametrize("mesh,nocc", [((1, 1, 2), 3), ((1, 1, 3), 8)])
def test_lane_sums_scale_and_pass_nan_on(mesh, nocc):
    """The contraction's sums over a warp's lanes (FP32: integers scaled by the largest lane):
    powers of two of C pass through every step exactly, zeros stay zeros and NaN stays NaN."""
    import torch
    import paper_2207_09028_gb300 as occri
    w = small_workload(mesh=mesh, grid=(12, 12, 12), counts=(5, 3), nocc=nocc, seed=53)
    plan = occri.Plan.from_workload(w, precision="mixed")
    C = torch.from_numpy(w.C).cuda()

    def kc(c):
        return plan.k_build(c, KC=torch.empty_like(c), sync=False)[0]

    ref = kc(C)
    for e in (-20, 9):
        assert torch.equal(kc(C * 2.0 ** e), ref * 2.0 ** (3 * e))
    zero = C.clone()
    zero[:, :, 1] = 0
    got = kc(zero)
    assert not got[:, :, 1].any() and torch.isfinite(torch.view_as_real(got)).all()
    for bad in (float("nan"), float("inf")):
        broken = C.clone()
        broken[0, 0, 0] = bad
        assert torch.isnan(torch.view_as_real(kc(broken))).all()
    with pytest.raises(occri.OccriError):   # (the zero and NaN builds are not positive definite)
        plan.sync()
    assert torch.equal(kc(C), ref)


def test_adjoint_of_a_tensor_core_plan():
    """The adjoint contracts on the CUDA cores in every plan: over items of their own."""
    import torch
    import paper_2207_09028_gb300 as occri
    w = small_workload(mesh=(1, 1, 2), grid=(12, 12, 12), counts=(2, 1), nocc=3, seed=45)
    G = torch.from_numpy(np.random.default_rng(6).standard_normal((w.nk, w.nao, w.nao)) + 0j).cuda()
    C = torch.from_numpy(w.C).cuda()
    out = {}
    for prec in ("fp64", "mixed_tc"):
        plan = occri.Plan.from_workload(w, precision=prec)
        plan.build(C)
        out[prec] = plan.vjp_full(C, 0.3, None, G).cpu().numpy()
    # the bar of the mixed adjoint: FP32 sums of about 2,000 points, 2000 u = 1.2e-4 at most,
    # sqrt(2000) u = 2.7e-6 as a random walk, with a margin of about 4
    assert np.abs(out["mixed_tc"] - out["fp64"]).max() <= 1e-5 * np.abs(out["fp64"]).max()
