"""When the defect correction stops: with room below refine_tol, after at most one pass that refine_tol did
not ask for, and never with a solution that meets refine_tol given up for a later one that does not."""
import numpy as np
import pytest

from paper_1801_08655_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def problem():
    from paper_1801_08655_gb300 import build, hz
    build.build()
    p = W.small_problem(26, 4, 4, seed=5, R=3)
    s = hz.Solver(p.m, p.omega, p.npml, p.C, p.n_layers, precision="mixed")
    s.factor()
    f = torch.from_numpy(p.rhs()).cuda()
    yield s, f
    s.close()


def solve(problem, tol, passes, gmres_tol=1e-5):
    from paper_1801_08655_gb300 import hz
    s, f = problem
    o = hz.default_opts("mixed")
    o.gmres_tol, o.refine_tol, o.max_refine = gmres_tol, tol, passes
    u, info, status = s.solve(f, o, allow_noconv=True)
    worst = max(i.volume_relres for i in info)
    again = max(s.volume_residual(f, u)[0])
    assert abs(again - worst) <= 1e-6 * worst   # the residual reported is the returned solution's
    return worst, info[0].refinements, status


def test_uncorrected_solution_needs_a_tenth(problem):
    from paper_1801_08655_gb300 import hz
    r0, n, _ = solve(problem, 1e-30, 0)
    assert n == 0
    assert solve(problem, 20 * r0, 3)[1] == 0             # a tenth: accepted as it is
    worst, n, status = solve(problem, 2 * r0, 3)          # between: corrected once
    assert n == 1 and status == hz.HZ_OK and worst < 0.5 * r0
    worst, n, status = solve(problem, 2 * r0, 0)          # met, and no pass allowed
    assert n == 0 and status == hz.HZ_OK
    assert solve(problem, 0.5 * r0, 0)[2] == hz.HZ_ERR_NO_CONVERGENCE


def test_tolerance_at_the_floor_of_the_residual(problem):
    """Once further passes no longer lower the residual, a tolerance just above that floor is met, and met
    with at most one pass more than it takes to get there."""
    from paper_1801_08655_gb300 import hz
    tail = [solve(problem, 1e-30, k)[0] for k in range(9)]
    floor = max(tail[4:])
    assert min(tail[4:]) > 0.4 * floor and tail[0] > 10 * floor   # flat, and far below the first pass
    tol = 1.2 * floor
    need = next(k for k in range(9) if tail[k] <= tol)
    worst, n, status = solve(problem, tol, 8)
    assert status == hz.HZ_OK and worst <= tol
    assert n <= need + 2, (n, need)   # one pass more where this run's passes differ by their rounding


def test_unreachable_tolerance_uses_its_passes(problem):
    from paper_1801_08655_gb300 import hz
    worst, n, status = solve(problem, 1e-30, 4)
    assert n == 4 and status == hz.HZ_ERR_NO_CONVERGENCE and np.isfinite(worst)


def test_solution_that_is_not_finite_is_not_converged(problem):
    """Sources beyond the range of the complex64 local solves: the residual is not a number, which no
    comparison with refine_tol may pass for converged."""
    from paper_1801_08655_gb300 import hz
    s, f = problem
    with pytest.raises(hz.HzError) as e:
        s.solve(f * 1e60, hz.default_opts("mixed"))
    assert e.value.status == hz.HZ_ERR_NONFINITE
    u = s.solve(f, hz.default_opts("mixed"))[0]           # the handle solves on
    assert bool(torch.isfinite(u.real).all())
