"""Correction steps on every level from one fine cell per half coarse cell up: the augmented step's
column segments end inside, at the end of and beyond the chunks a thread walks, are empty or are cut
off by the boundary.

FP64: the oracle's step, from the same iterate, to 1e-12 of the solution (its dense systems have
condition numbers below 1e3, their assembly and solution a few hundred roundings of 1e-16).  Mixed: the
iterate stays float-float and the corrections to it are FP32, which the Newton test at 1e-6 ends: 1e-6."""
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


@pytest.mark.parametrize("nonlinear", ["newton", "fixed_point"])
@pytest.mark.parametrize("dim,H,r", [(2, 2, 8), (2, 6, 5), (2, 8, 5), (3, 2, 5), (3, 4, 3)])
def test_correction_step_on_every_level(fmg, dim, H, r, nonlinear):
    prob = W.Problem(dim=dim, coarse_cells=H, refinements=r, f="cubic",
                     modes=[((1,) * dim, 1.0), ((2,) + (1,) * (dim - 1), 0.6)])
    g = prob.g_nodal()
    hier = O.build_hierarchy(dim, H, r)
    solvers = {p: fmg.Solver(fmg.make_params(prob, precision=p, smoother="rbgs", nonlinear=nonlinear), g)
               for p in ("fp64", "mixed")}
    rng = np.random.default_rng(10 * dim + H)
    for k in range(2, r + 2):
        lev = hier.level(k)
        gk = O.restrict_nodal(g, dim, H << r, lev.n)
        us = O.from_nodal(lev, O.restrict_nodal(prob.u_star(), dim, H << r, lev.n))
        U = us * (1.0 + 0.05 * rng.standard_normal(len(us)))
        want, _ = O.correction_step(hier, k, U, O.load_vector(lev, gk), prob.f, prob.a, nonlinear=nonlinear)
        for p, tol in (("fp64", 1e-12), ("mixed", 1e-6)):
            u = torch.tensor(O.to_nodal(lev, U), device="cuda")
            fmg.fmg_op_correction_step(solvers[p].ctx, k, u)
            got = O.from_nodal(lev, u.cpu().numpy())
            assert np.max(np.abs(got - want)) <= tol * np.max(np.abs(want)), (k, p)
    for s in solvers.values():
        s.close()
