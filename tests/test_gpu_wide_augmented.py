"""The correction step of contexts that run side by side (batches, the request server) on levels
large enough for the wide form (fine passes as launches over the whole device, the last block taking
the dense step, the cluster kernel doing what is left) against the same solve alone.

The two forms differ in the order of the block sums only.  FP64: the FP64 bar.  Mixed: the sums are
float-float (2^-44) and the chord steps contract, so a Newton iteration stopped at tol leaves the
two solves apart by rounding and by at most the last step's contraction of tol = 1e-6, a few 1e-9 of
the solution; the bar is 1e-8.  1/H = 2 reaches the wide form at the smallest sizes (a cluster
of 4 or 8 CTAs).
"""
import numpy as np
import pytest

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


def problem(dim, H, r, f):
    modes = [((1,) * dim, 1.0), ((2,) + (1,) * (dim - 1), 0.3)]
    return W.Problem(dim=dim, coarse_cells=H, refinements=r, f=f, a=1.0, modes=modes)


# Newton options: the defaults, one iteration only, a tolerance that takes more than two, and the
# fixed-point iteration
OPTIONS = [{}, {"newton_maxit": 1}, {"newton_tol": 1e-10}, {"nonlinear": 1}]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("dim,H,r,f", [(2, 2, 7, "cubic"), (2, 2, 8, "linear"), (2, 4, 7, "expm1"),
                                       (2, 8, 6, "signed_pow32"), (3, 2, 4, "cubic"), (3, 4, 4, "expm1"),
                                       (3, 4, 5, "neg_exp_neg")])
def test_batch_equals_solo(fmg, dim, H, r, f, precision):
    p = problem(dim, H, r, f)
    g = p.g_nodal()
    for opt in OPTIONS if r + dim < 9 else OPTIONS[:1]:
        solvers = [fmg.Solver(fmg.make_params(p, precision=precision, **opt), g) for _ in range(2)]
        st = fmg.fmg_stats()
        try:
            solo = solvers[0].solve(stats=st).cpu().numpy()
        except fmg.FMGError as e:   # one iteration does not converge: the batch has to say so too
            with pytest.raises(fmg.FMGError) as got:
                fmg.Batch(solvers).solve(wait=True)
            assert got.value.status == e.status
            continue
        batch = fmg.Batch(solvers)
        stats = batch.solve(wait=True)
        bar = 1e-10 if precision == "fp64" else 1e-8
        first = solvers[0].solution().cpu().numpy()
        assert np.max(np.abs(first - solo)) <= bar * np.max(np.abs(solo)), opt
        assert np.array_equal(first, solvers[1].solution().cpu().numpy())
        for k in range(r + 1):
            assert abs(stats[0].newton_iters[k] - st.newton_iters[k]) <= 1, (k, opt)
        batch.solve(wait=True)
        assert np.array_equal(first, solvers[0].solution().cpu().numpy())
        batch.close()
