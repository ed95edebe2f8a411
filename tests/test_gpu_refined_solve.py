"""The linear solves of the FP64 Newton steps, which refine on an FP32 inverse, on problems whose
solution is small: the coarse values then lie far below alpha, which stays near 1.

Level 1 against the exact solution of the discrete system in extended precision: the solve is backward
stable, so its error is at most the condition number of A_1 (26 at 1/H = 8) times the rounding of
a row's nine operations, 26 * 9 * 1.1e-16 = 2.6e-14 of the maximum.  Correction steps and solves
against the oracle at the FP64 bar of 1e-10 relative to the solution, whatever its size."""
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


def problem(dim, H, r, f, amp):
    return W.Problem(dim=dim, coarse_cells=H, refinements=r, f=f,
                     modes=[((1,) * dim, amp), ((2,) + (1,) * (dim - 1), 0.35 * amp)])


def extended_solve(A, b):
    """A x = b by elimination in extended precision (A symmetric positive definite)."""
    A, b = A.astype(np.longdouble), b.astype(np.longdouble)
    n = len(b)
    for k in range(n):
        m = A[k + 1:, k] / A[k, k]
        A[k + 1:, k:] -= np.outer(m, A[k, k:])
        b[k + 1:] -= m * b[k]
    x = np.zeros(n, dtype=np.longdouble)
    for k in range(n - 1, -1, -1):
        x[k] = (b[k] - A[k, k + 1:] @ x[k + 1:]) / A[k, k]
    return x


@pytest.mark.parametrize("amp", [1.0, 1e-9, 1e-15])
@pytest.mark.parametrize("dim,H", [(2, 4), (2, 6), (2, 8), (3, 4)])
def test_level1_small_solution(fmg, dim, H, amp):
    """f(u) = a u: the level-1 system is linear."""
    prob = problem(dim, H, 1, "linear", amp)
    g = prob.g_nodal()
    lev = O.build_hierarchy(dim, H, 0).level(1)
    G = O.load_vector(lev, O.restrict_nodal(g, dim, 2 * H, H))
    A = lev.A.toarray() + np.diag(prob.a * lev.w * np.ones(len(G)))
    ref = extended_solve(A, G)
    s = fmg.Solver(fmg.make_params(prob, precision="fp64"), g)
    u = torch.zeros((H + 1,) * dim, dtype=torch.float64, device="cuda")
    fmg.fmg_op_level1_solve(s.ctx, u)
    s.close()
    got = O.from_nodal(lev, u.cpu().numpy())
    assert np.max(np.abs(got - ref)) <= 2.6e-14 * np.max(np.abs(ref))


@pytest.mark.parametrize("f", ["cubic", "linear"])
@pytest.mark.parametrize("amp", [1e-6, 1e-9, 1e-12])
@pytest.mark.parametrize("dim,H,r", [(2, 4, 3), (2, 8, 3), (3, 4, 2)])
def test_small_solution(fmg, dim, H, r, amp, f):
    prob = problem(dim, H, r, f, amp)
    g = prob.g_nodal()
    hier = O.build_hierarchy(dim, H, r)
    lev = hier.level(r + 1)
    ref = O.to_nodal(lev, O.fmg(hier, g, prob.f, prob.a).u[-1])
    s = fmg.Solver(fmg.make_params(prob, precision="fp64"), g)
    got = s.solve().cpu().numpy()
    assert np.max(np.abs(got - ref)) <= 1e-10 * np.max(np.abs(ref))
    # a correction step from an iterate a tenth off
    rng = np.random.default_rng(5)
    U = O.from_nodal(lev, ref) * (1.0 + 0.1 * rng.standard_normal(lev.A.shape[0]))
    want = O.to_nodal(lev, O.correction_step(hier, r + 1, U, O.load_vector(lev, g), prob.f, prob.a)[0])
    u = torch.tensor(O.to_nodal(lev, U), device="cuda")
    fmg.fmg_op_correction_step(s.ctx, r + 1, u)
    s.close()
    assert np.max(np.abs(u.cpu().numpy() - want)) <= 1e-10 * np.max(np.abs(want))


def iterations(hier, k, ut, G, f, a, count, fixed_point):
    """`count` iterations of (3.6) from (c, alpha) = (0, 1), in FP64 with a dense factorization."""
    lev = hier.level(k)
    B = np.hstack([hier.P_H[k - 1].toarray(), ut[:, None]])
    K = B.T @ (lev.A @ B)
    y = np.zeros(B.shape[1])
    y[-1] = 1.0
    for _ in range(count):
        U = B @ y
        R = K @ y + B.T @ (lev.w * O.f_val(f, a, U) - G)
        J = K if fixed_point else K + B.T @ ((lev.w * O.f_der(f, a, U))[:, None] * B)
        d = np.linalg.solve(J, R)
        y = y - d
        if np.max(np.abs(d)) <= 1e-6 * max(1.0, np.max(np.abs(y))):
            break
    return B @ y


@pytest.mark.parametrize("nonlinear", ["newton", "fixed_point"])
@pytest.mark.parametrize("count", [1, 2, 3])
@pytest.mark.parametrize("dim,H,r", [(2, 4, 3), (2, 8, 3), (3, 4, 2)])
def test_iteration_cut_short(fmg, dim, H, r, count, nonlinear):
    """The iterate after any number of steps is that of steps solved in FP64, whose dense solves have
    errors of up to 3e-13 on these systems: 1e-12 of the solution."""
    prob = problem(dim, H, r, "cubic", 2.0)
    g = prob.g_nodal()
    hier = O.build_hierarchy(dim, H, r)
    lev = hier.level(r + 1)
    G = O.load_vector(lev, g)
    rng = np.random.default_rng(6)
    U = O.from_nodal(lev, prob.u_star()) * (1.0 + 0.5 * rng.standard_normal(lev.A.shape[0]))
    b = G - lev.w * O.f_val(prob.f, prob.a, U)
    ut = U.copy()
    for _ in range(2):
        ut = O.vcycle(hier, r + 1, b, ut, 2, 2)
    want = O.to_nodal(lev, iterations(hier, r + 1, ut, G, prob.f, prob.a, count, nonlinear == "fixed_point"))
    s = fmg.Solver(fmg.make_params(prob, precision="fp64", nonlinear=nonlinear, newton_maxit=count), g)
    u = torch.tensor(O.to_nodal(lev, U), device="cuda")
    try:
        fmg.fmg_op_correction_step(s.ctx, r + 1, u)
    except fmg.FMGError:
        pass   # (the cap is reported)
    got = u.cpu().numpy()
    s.close()
    assert np.max(np.abs(got - want)) <= 1e-12 * np.max(np.abs(want))
