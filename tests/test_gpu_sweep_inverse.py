"""The dense systems of the Newton steps at every size the solver takes (1/H = 2 to 8 in 2D, 2 and 4 in
3D: 2, 10, 26, 50 and 2, 28 unknowns, one less at level 1), whose FP32 inverse the block-wide sweep forms.

FP64 path against the oracle at the FP64 bar.  Mixed path against the FP64 one: the iterations stop at
tol = 1e-6 and contract, and the cycles are FP32 corrections of float-float residuals, so the two
stay within 1e-7 of the solution.
"""
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


@pytest.mark.parametrize("f", ["cubic", "neg_exp_neg"])
@pytest.mark.parametrize("dim,H", [(2, 2), (2, 4), (2, 6), (2, 8), (3, 2), (3, 4)])
def test_every_coarse_size(fmg, dim, H, f):
    prob = W.Problem(dim=dim, coarse_cells=H, refinements=2, f=f, modes=[((1,) * dim, 2.0), ((2,) + (1,) * (dim - 1), 0.7)])
    g = prob.g_nodal()
    hier = O.build_hierarchy(dim, H, 2)
    ref = O.to_nodal(hier.level(3), O.fmg(hier, g, prob.f, prob.a).u[-1])
    scale = np.max(np.abs(ref))
    got = fmg.Solver(fmg.make_params(prob, precision="fp64"), g).solve().cpu().numpy()
    assert np.max(np.abs(got - ref)) <= 1e-10 * scale
    mixed = fmg.Solver(fmg.make_params(prob, precision="mixed", smoother="rbgs"), g).solve().cpu().numpy()
    assert np.max(np.abs(mixed - got)) <= 1e-7 * scale
