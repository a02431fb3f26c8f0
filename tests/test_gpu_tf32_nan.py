"""A NaN in one column of the preconditioner's input reaches that column's whole result, and no other's,
through the tensor-core substitutions with three TF32 terms and with the single-term option."""
import pytest

from paper_1801_08655_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split", ["1", "3"])
@pytest.mark.parametrize("cfg", ["0", "1"])
@pytest.mark.parametrize("R", [32, 64, 128])
def test_nan_goes_through_the_preconditioner(R, cfg, split, monkeypatch):
    from paper_1801_08655_gb300 import build, hz
    build.build()
    for k, v in (("HZ_SUBST_TC", "1"), ("HZ_TC_MIN_TILES", "1"), ("HZ_AUTOTUNE", "0"), ("HZ_TC_CFG", cfg),
                 ("HZ_PRECOND_SPLIT", split)):
        monkeypatch.setenv(k, v)
    p = W.small_problem(26, 4, 4, seed=5, R=1)
    s = hz.Solver(p.m, p.omega, p.npml, p.C, p.n_layers, precision="mixed")
    s.factor()
    g = torch.Generator("cuda").manual_seed(R)
    x = torch.randn(s.trace_shape(R), dtype=torch.complex128, device="cuda", generator=g)
    x[5, 0, 0, 1, 7, 9] = complex(float("nan"), float("nan"))   # down-going, first interface, its layer-1 plane
    y = s.apply_precond(x)
    bad = torch.isnan(y.real) | torch.isnan(y.imag)
    assert bool(bad[5, 0, 1:].all())                            # solved on from the first interface
    assert not bool(bad[:5].any()) and not bool(bad[6:].any())
    s.close()
