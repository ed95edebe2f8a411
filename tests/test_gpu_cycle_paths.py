"""Forms of the cycle kernels that the default settings do not reach: the dealt 2D cycle's exchange in
the middle of a level's smoothing (more than three red-black sweeps, six Chebyshev steps; with the
step direction from seven), the FP64 tile kernels with one sweep and with unequal counts, the
no-allocation cycle on every mesh of the tile kernels, the float-float update of a dealt top level,
and the FP64 factorization behind the refined solves.

FP64 cycles against the oracle's to 1e-12 (a few hundred roundings of 1e-16 relative to the
iterate), mixed ones to 1e-4 (the same of 6e-8 relative to a correction no larger than the iterate)."""
import functools

import numpy as np
import pytest

from oracle import fmg_oracle as O
from paper_1611_05677_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def fmg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    from paper_1611_05677_gb300 import fmg as F

    F.load()
    return F


@functools.lru_cache(maxsize=None)
def linear_problem(dim, H, r):
    hier = O.build_hierarchy(dim, H, r)
    lev = hier.level(r + 1)
    n = H << r
    rng = np.random.default_rng(7 * n + dim)
    b = O.to_nodal(lev, rng.standard_normal((n - 1) ** dim) / n ** dim)
    u0 = O.to_nodal(lev, 0.1 * rng.standard_normal((n - 1) ** dim))
    return hier, lev, b, u0


def oracle_cycles(hier, lev, k, b, u0, nu, smoother, cycles):
    u = O.from_nodal(lev, u0).copy()
    for _ in range(cycles):
        u = O.vcycle(hier, k, O.from_nodal(lev, b), u, nu[0], nu[1], smoother)
    return O.to_nodal(lev, u)


def cycles_of(fmg, dim, H, r, precision, smoother, nu, cycles=2):
    hier, lev, b, u0 = linear_problem(dim, H, r)
    prob = W.Problem(dim=dim, coarse_cells=H, refinements=r, modes=[((1,) * dim, 1.0)])
    s = fmg.Solver(fmg.make_params(prob, precision=precision, smoother=smoother, nu_pre=nu[0], nu_post=nu[1]),
                   np.zeros(b.shape))
    u = torch.tensor(u0, device="cuda")
    fmg.fmg_op_vcycle(s.ctx, r + 1, torch.tensor(b, device="cuda"), u, cycles)
    got = u.cpu().numpy()
    s.close()
    return got, oracle_cycles(hier, lev, r + 1, b, u0, nu, smoother, cycles)


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("mixed", 1e-4)])
@pytest.mark.parametrize("smoother,nu", [("rbgs", (4, 5)), ("rbgs", (9, 0)), ("rbgs", (0, 7)), ("chebyshev", (7, 6)),
                                         ("chebyshev", (8, 13)), ("chebyshev", (16, 16))])
@pytest.mark.parametrize("H,r", [(8, 3), (6, 3), (4, 5)])
def test_many_sweeps_on_dealt_rows(fmg, H, r, smoother, nu, precision, tol):
    """(4, 5): 128 cells, the dealt level below the top one."""
    got, ref = cycles_of(fmg, 2, H, r, precision, smoother, nu)
    assert np.max(np.abs(got - ref)) <= tol * np.max(np.abs(ref))


@pytest.mark.parametrize("smoother,nu", [("rbgs", (5, 4)), ("chebyshev", (16, 7))])
def test_many_sweeps_on_dealt_planes(fmg, smoother, nu):
    got, ref = cycles_of(fmg, 3, 4, 2, "fp64", smoother, nu)
    assert np.max(np.abs(got - ref)) <= 1e-12 * np.max(np.abs(ref))


@pytest.mark.parametrize("nu", [(1, 1), (1, 2), (2, 1), (3, 1), (2, 0), (0, 2)])
@pytest.mark.parametrize("H,r", [(4, 5), (6, 4), (4, 6), (8, 6)])
def test_tile_kernel_sweeps(fmg, H, r, nu):
    """128, 96, 256 and 512 cells."""
    got, ref = cycles_of(fmg, 2, H, r, "fp64", "rbgs", nu)
    assert np.max(np.abs(got - ref)) <= 1e-12 * np.max(np.abs(ref))


@pytest.mark.parametrize("nu", [(2, 2), (1, 1), (2, 1), (3, 3), (0, 2), (1, 0)])
@pytest.mark.parametrize("dim,H,level", [(2, 4, 7), (2, 8, 7), (2, 6, 6), (3, 4, 4)])
def test_noalloc_sweeps(fmg, dim, H, level, nu):
    hier, lev, b, u0 = linear_problem(dim, H, level - 1)
    u = torch.tensor(u0, device="cuda")
    stream = torch.cuda.Stream()
    bd = torch.tensor(b, device="cuda")
    torch.cuda.synchronize()
    fmg.fmg_vcycle_noalloc(dim, H, level, bd, u, cycles=2, nu_pre=nu[0], nu_post=nu[1], stream=stream)
    stream.synchronize()
    ref = oracle_cycles(hier, lev, level, b, u0, nu, "rbgs", 2)
    assert np.max(np.abs(u.cpu().numpy() - ref)) <= 1e-12 * np.max(np.abs(ref))


@pytest.mark.parametrize("smoother", ["rbgs", "chebyshev"])
@pytest.mark.parametrize("dim,H,k", [(2, 8, 4), (2, 6, 4), (3, 4, 3)])
def test_float_float_update_of_a_dealt_top_level(fmg, dim, H, k, smoother):
    """A correction step on 64^2, 48^2 and 16^3 cells from an iterate 1e-4 off: the corrections are at
    most 1e-3 of it and carry FP32 rounding of a cycle, 1e-6; 1e-8 in all is below a third of the
    6e-8 that a lost low word would leave."""
    prob = W.Problem(dim=dim, coarse_cells=H, refinements=k - 1, f="cubic", modes=[((1,) * dim, 1.0)])
    g = prob.g_nodal()
    hier = O.build_hierarchy(dim, H, k - 1)
    lev = hier.level(k)
    sol = O.fmg(hier, g, prob.f, prob.a, smoother=smoother).u[-1]
    U = sol * (1.0 + 1e-4 * np.random.default_rng(3).standard_normal(len(sol)))
    want, _ = O.correction_step(hier, k, U, O.load_vector(lev, g), prob.f, prob.a, smoother=smoother)
    s = fmg.Solver(fmg.make_params(prob, precision="mixed", smoother=smoother), g)
    u = torch.tensor(O.to_nodal(lev, U), device="cuda")
    fmg.fmg_op_correction_step(s.ctx, k, u)
    s.close()
    assert np.max(np.abs(O.from_nodal(lev, u.cpu().numpy()) - want)) <= 1e-8 * np.max(np.abs(want))


@pytest.mark.parametrize("dim,H,r", [(2, 4, 3), (2, 8, 3), (3, 4, 2)])
def test_factorization_when_the_iterate_is_almost_coarse(fmg, dim, H, r):
    """The level's solution is a coarse function up to 1e-3: the Schur complement of alpha is below
    the 1e-3 of its diagonal that the FP32 inverse asks for, so the step is solved in FP64.  The
    system's condition number is 3e4 to 3e5: 1e-10 in u at most."""
    hier = O.build_hierarchy(dim, H, r)
    k = r + 1
    lev = hier.level(k)
    rng = np.random.default_rng(11)
    x = np.linspace(0, 1, H + 1)
    bump = np.ones((1,))
    for _ in range(dim):
        bump = np.multiply.outer(np.sin(np.pi * x), bump)
    coarse = hier.P_H[k - 1] @ O.from_nodal(hier.level(1), bump[..., 0])
    a = 1.0
    us = coarse * (1.0 + 1e-3 * rng.standard_normal(len(coarse)))
    G = lev.A @ us + lev.w * O.f_val("cubic", a, us)
    g = O.to_nodal(lev, G / lev.w)
    U = us * (1.0 + 1e-3 * rng.standard_normal(len(us)))
    want, info = O.correction_step(hier, k, U, G, "cubic", a)
    prob = W.Problem(dim=dim, coarse_cells=H, refinements=r, f="cubic", modes=[((1,) * dim, 1.0)])
    s = fmg.Solver(fmg.make_params(prob, precision="fp64"), g)
    u = torch.tensor(O.to_nodal(lev, U), device="cuda")
    fmg.fmg_op_correction_step(s.ctx, k, u)
    s.close()
    assert np.max(np.abs(O.from_nodal(lev, u.cpu().numpy()) - want)) <= 1e-10 * np.max(np.abs(want))


def test_factorization_of_level1_below_fp32(fmg):
    """A solution of 1e-25, which leaves FP32 no room for the refinement: proportional to the
    one of a load 2^80 times as large."""
    prob = W.Problem(dim=2, coarse_cells=8, refinements=1, f="linear", modes=[((1, 1), 1.0), ((2, 1), 0.4)])
    g = prob.g_nodal()
    out = []
    for scale in (1.0, 2.0 ** -80):
        s = fmg.Solver(fmg.make_params(prob, precision="fp64"), g * scale)
        u = torch.zeros((9, 9), dtype=torch.float64, device="cuda")
        fmg.fmg_op_level1_solve(s.ctx, u)
        s.close()
        out.append(u.cpu().numpy() / scale)
    assert np.max(np.abs(out[0] - out[1])) <= 1e-13 * np.max(np.abs(out[0]))
