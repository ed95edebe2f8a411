"""V-cycles whose levels run in the cluster coarse-cycle kernel, alone and below the per-level
kernels, against the oracle's V-cycle: every mesh the kernel deals to its CTAs differently (fewer
rows than CTAs, one row each, several, 1/H that is no power of two), both smoothers, sweep counts
down to zero, a variable coefficient, and the float-float and FP64 updates of the mixed path.

Tolerances: a cycle's FP64 rounding error is a few hundred operations' 1e-16 relative to the
iterate, and the red-black form leaves out residuals that are zero but for that rounding, so
1e-12.  A mixed cycle's correction carries FP32 rounding, a few hundred 6e-8 relative to itself,
and is no larger than the iterate, so 1e-4."""
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


SHAPES = [(2, 2, 1), (2, 2, 6), (2, 4, 4), (2, 6, 3), (2, 6, 4), (2, 8, 1), (2, 8, 3), (2, 8, 4),
          (3, 2, 1), (3, 2, 3), (3, 4, 1), (3, 4, 2), (3, 4, 3)]


def cycle_pair(fmg, dim, H, r, precision, smoother, nu, coef=None, cycles=2):
    hier = O.build_hierarchy(dim, H, r, coef=coef)
    lev = hier.level(r + 1)
    n = H << r
    rng = np.random.default_rng(100 * dim + 10 * H + r)
    b = O.to_nodal(lev, rng.standard_normal((n - 1) ** dim) / n ** dim)
    u0 = O.to_nodal(lev, 0.1 * rng.standard_normal((n - 1) ** dim))
    ref = O.from_nodal(lev, u0).copy()
    for _ in range(cycles):
        ref = O.vcycle(hier, r + 1, O.from_nodal(lev, b), ref, nu[0], nu[1], smoother)
    prob = W.Problem(dim=dim, coarse_cells=H, refinements=r, modes=[((1,) * dim, 1.0)], coefficient=coef)
    s = fmg.Solver(fmg.make_params(prob, precision=precision, smoother=smoother, nu_pre=nu[0], nu_post=nu[1]),
                   np.zeros((n + 1,) * dim))
    u = torch.tensor(u0, device="cuda")
    fmg.fmg_op_vcycle(s.ctx, r + 1, torch.tensor(b, device="cuda"), u, cycles)
    got = u.cpu().numpy()
    s.close()
    return got, O.to_nodal(lev, ref)


@pytest.mark.parametrize("smoother", ["rbgs", "chebyshev"])
@pytest.mark.parametrize("dim,H,r", SHAPES)
def test_fp64_cycle(fmg, dim, H, r, smoother):
    got, ref = cycle_pair(fmg, dim, H, r, "fp64", smoother, (2, 2))
    assert np.max(np.abs(got - ref)) <= 1e-12 * np.max(np.abs(ref))


@pytest.mark.parametrize("smoother", ["rbgs", "chebyshev"])
@pytest.mark.parametrize("nu", [(1, 0), (0, 1), (3, 1), (1, 2)])
@pytest.mark.parametrize("dim,H,r", [(2, 8, 3), (2, 6, 2), (3, 4, 2)])
def test_fp64_cycle_sweeps(fmg, dim, H, r, nu, smoother):
    got, ref = cycle_pair(fmg, dim, H, r, "fp64", smoother, nu)
    assert np.max(np.abs(got - ref)) <= 1e-12 * np.max(np.abs(ref))


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("mixed", 1e-4)])
@pytest.mark.parametrize("dim,H,r", [(2, 8, 3), (2, 6, 4), (2, 2, 2), (3, 4, 2), (3, 2, 3)])
def test_coefficient_cycle(fmg, dim, H, r, precision, tol):
    got, ref = cycle_pair(fmg, dim, H, r, precision, "rbgs", (2, 2), coef=W.cell_coefficient(dim, H))
    assert np.max(np.abs(got - ref)) <= tol * np.max(np.abs(ref))


@pytest.mark.parametrize("smoother", ["rbgs", "chebyshev"])
@pytest.mark.parametrize("dim,H,r", SHAPES)
def test_mixed_cycle(fmg, dim, H, r, smoother):
    got, ref = cycle_pair(fmg, dim, H, r, "mixed", smoother, (2, 2))
    assert np.max(np.abs(got - ref)) <= 1e-4 * np.max(np.abs(ref))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_solve_with_six_coarse_cells(fmg, precision):
    """1/H = 6: coarse meshes of 6, 12, 24 and 48 cells per side."""
    prob = W.Problem(dim=2, coarse_cells=6, refinements=4, f="cubic", modes=[((1, 2), 1.0), ((3, 1), 0.5)])
    g = prob.g_nodal()
    hier = O.build_hierarchy(2, 6, 4)
    ref = O.to_nodal(hier.level(5), O.fmg(hier, g, prob.f, prob.a).u[-1])
    s = fmg.Solver(fmg.make_params(prob, precision=precision), g)
    got = s.solve().cpu().numpy()
    s.close()
    disc = np.max(np.abs(ref - prob.u_star()))
    tol = 1e-10 * np.max(np.abs(ref)) if precision == "fp64" else 0.1 * disc
    assert np.max(np.abs(got - ref)) <= tol
