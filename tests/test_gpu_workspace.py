"""A caller's workspace may start at any address (fmg_create): the arrays that the kernels read in
16-byte words start on aligned addresses inside it, and a solve gives the bits it gives elsewhere."""
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


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("dim,H,r", [(2, 4, 3), (3, 2, 3)])
def test_workspace_at_any_address(fmg, dim, H, r, precision):
    prob = W.Problem(dim=dim, coarse_cells=H, refinements=r, f="cubic", modes=[((1,) * dim, 1.0)])
    g = prob.g_nodal()
    params = fmg.make_params(prob, precision=precision)
    need = fmg.fmg_workspace_bytes(params)
    ref = fmg.Solver(params, g).solve().cpu().numpy()
    stream = torch.cuda.Stream()
    for off in (0, 1, 8, 16, 24, 255):
        memory = torch.zeros(need + 256, dtype=torch.uint8, device="cuda")
        part = memory[off:off + need]
        torch.cuda.synchronize()
        ctx = fmg.fmg_create(params, g, stream.cuda_stream, part, need)
        first = fmg.fmg_solution(ctx)
        assert first % 256 == 0 and part.data_ptr() <= first < part.data_ptr() + need
        u = torch.empty(ref.shape, dtype=torch.float64, device="cuda")
        fmg.fmg_solve(ctx, u)
        stream.synchronize()
        assert np.array_equal(u.cpu().numpy(), ref), off
        fmg.fmg_destroy(ctx)
        # nothing before or behind the part was written
        assert int(memory[:off].sum()) == 0 and int(memory[off + need:].sum()) == 0


def test_short_workspace_is_refused(fmg):
    prob = W.Problem(dim=2, coarse_cells=4, refinements=3, f="cubic", modes=[((1, 1), 1.0)])
    params = fmg.make_params(prob, precision="fp64")
    need = fmg.fmg_workspace_bytes(params)
    memory = torch.zeros(need, dtype=torch.uint8, device="cuda")
    with pytest.raises(fmg.FMGError) as ei:
        fmg.fmg_create(params, prob.g_nodal(), torch.cuda.Stream().cuda_stream, memory, need - 1)
    assert ei.value.status == fmg.FMG_ERR_INVALID
