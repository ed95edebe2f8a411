"""V-cycles whose top level is a 16^3 mesh dealt to the CTAs of a cluster with a halo of one plane:
the exchanges of the planes between CTAs that are not in step.

After the prolongation a CTA has added the correction to its halo planes in place; a neighbour's
plane that arrived before that would be corrected twice.  After an odd number of Chebyshev steps
from a given iterate the result is moved to the buffer that the last step read; a plane of it that
arrived in a neighbour still in that step would take the old one's place.  Every run has the same arithmetic in the
same order, so many runs from one start give one set of bits, and those are the oracle's cycle to
1e-12 (a few hundred FP64 operations' rounding relative to the iterate; 1e-4 for the FP32 cycles)."""
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


def repeated_cycles(fmg, H, r, precision, smoother, nu, coef=None, runs=60, cycles=2):
    hier = O.build_hierarchy(3, H, r, coef=coef)
    lev = hier.level(r + 1)
    n = H << r
    rng = np.random.default_rng(30 + 10 * H + r)
    b = O.to_nodal(lev, rng.standard_normal((n - 1) ** 3) / n ** 3)
    u0 = O.to_nodal(lev, 0.1 * rng.standard_normal((n - 1) ** 3))
    ref = O.from_nodal(lev, u0).copy()
    for _ in range(cycles):
        ref = O.vcycle(hier, r + 1, O.from_nodal(lev, b), ref, nu[0], nu[1], smoother)
    ref = O.to_nodal(lev, ref)
    prob = W.Problem(dim=3, coarse_cells=H, refinements=r, modes=[((1, 1, 1), 1.0)], coefficient=coef)
    s = fmg.Solver(fmg.make_params(prob, precision=precision, smoother=smoother, nu_pre=nu[0], nu_post=nu[1]),
                   np.zeros((n + 1,) * 3))
    bd, ud = torch.tensor(b, device="cuda"), torch.tensor(u0, device="cuda")
    first = None
    for _ in range(runs):
        u = ud.clone()
        torch.cuda.synchronize()
        fmg.fmg_op_vcycle(s.ctx, r + 1, bd, u, cycles)
        got = u.cpu().numpy()
        if first is None:
            first = got
        assert np.array_equal(got, first)
    s.close()
    tol = 1e-12 if precision == "fp64" else 1e-4
    assert np.max(np.abs(first - ref)) <= tol * np.max(np.abs(ref))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("nu", [(2, 2), (1, 1), (0, 3)])
@pytest.mark.parametrize("H,r", [(4, 2), (2, 3)])
def test_red_black_after_prolongation(fmg, H, r, nu, precision):
    repeated_cycles(fmg, H, r, precision, "rbgs", nu)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_red_black_after_prolongation_with_coefficient(fmg, precision):
    repeated_cycles(fmg, 4, 2, precision, "rbgs", (1, 2), coef=W.cell_coefficient(3, 4))


@pytest.mark.parametrize("nu", [(1, 1), (3, 0), (5, 2), (2, 3)])
@pytest.mark.parametrize("H,r", [(4, 2), (2, 3)])
def test_odd_chebyshev_steps(fmg, H, r, nu):
    repeated_cycles(fmg, H, r, "fp64", "chebyshev", nu)
