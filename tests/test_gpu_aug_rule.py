"""The default launch shape of the augmented kernel is one of those that fmg_autotune_augmented times
(chunks of 2 to 32 fine nodes, a power of two within the column), so that tuning never keeps a shape
slower than the default."""
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


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("dim,H,r", [(2, 2, 8), (2, 4, 6), (2, 6, 5), (2, 8, 6), (3, 2, 5), (3, 4, 4)])
def test_default_shape_is_a_candidate(fmg, dim, H, r, precision):
    prob = W.Problem(dim=dim, coarse_cells=H, refinements=r, f="cubic", modes=[((1,) * dim, 1.0)])
    s = fmg.Solver(fmg.make_params(prob, precision=precision), prob.g_nodal())
    for k in range(2, r + 2):
        chunk, bpc = fmg.fmg_aug_shape(s.ctx, k)
        assert chunk in (2, 4, 8, 16, 32) and chunk <= 1 << (k - 1), (k, chunk)
        assert bpc >= 1
    s.close()
