"""Complex64 local solves on M21 = L21 L11^{-1} against the CPU oracle's operator, on boxes and tree
shapes where tiles are ragged: one-node trees, nodes of one tile, fronts on either side of the
tensor-core threshold.  Tolerance: the mixed-precision stage tolerance (2e-4 relative, FP32
rounding through an unpivoted LDL^T)."""
import numpy as np
import pytest
import scipy.sparse.linalg as spla

from oracle import discretization as D
from paper_1801_08655_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def solve_and_compare(s, shape, m, omega, npml, C, cols, rng):
    nz, ny, nx = shape
    A = D.assemble(m, omega, *[D.global_profiles(n, npml, C, omega) for n in (nx, ny, nz)]).tocsc()
    lu = spla.splu(A)
    for R in cols:
        g = rng.standard_normal((R,) + shape) + 1j * rng.standard_normal((R,) + shape)
        ref = lu.solve(np.ascontiguousarray(g.reshape(R, -1).T)).T.reshape(g.shape)
        w = s.layer_solve(0, torch.from_numpy(g).cuda()).cpu().numpy()
        err = np.linalg.norm(w - ref) / np.linalg.norm(ref)
        assert err < 2e-4, (R, err)


@pytest.mark.parametrize("shape,leaf,tc_min,cols", [
    ((4, 5, 7), 1000, 128, (1, 3)),        # a single node of 140 unknowns: no update rows
    ((3, 4, 9), 8, 1, (2,)),               # nodes of a few cells
    ((9, 33, 10), 64, 128, (1, 17, 64)),   # ragged tiles, panel-step fronts only
    ((21, 24, 23), 256, 1, (1, 33, 64, 128)),   # every front of a tile or more on the tensor cores
    ((21, 24, 23), 256, 0, (5, 64)),       # none
])
@pytest.mark.parametrize("precision", ["mixed", "mixed64"])
def test_layer_solve_on_m21(shape, leaf, tc_min, cols, precision, monkeypatch):
    from paper_1801_08655_gb300 import build, hz
    build.build()
    monkeypatch.setenv("HZ_LEAF", str(leaf))
    monkeypatch.setenv("HZ_FACTOR_TC_MIN", str(tc_min))
    nz, ny, nx = shape
    rng = np.random.default_rng(nx + ny + nz)
    c = 1.5 + rng.random(shape)
    m, omega, npml, C = 1.0 / (c * c), W.omega_for_ppw(1.5, 9.0), 1, W.pml_constant(2.5)
    s = hz.Solver(m, omega, npml, C, 1, precision=precision)
    s.factor()
    solve_and_compare(s, shape, m, omega, npml, C, cols, rng)
    s.close()


@pytest.mark.parametrize("shape", [(21, 24, 23), (9, 33, 10)])
@pytest.mark.parametrize("cfg", [0, 1])
def test_narrow_column_blocks_on_the_tensor_cores(shape, cfg, monkeypatch):
    """17 to 128 columns (tiles of 32, 64 and 128) forced onto the tensor-core kernels."""
    from paper_1801_08655_gb300 import build, hz
    build.build()
    for k, v in (("HZ_SUBST_TC", 1), ("HZ_TC_MIN_TILES", 2), ("HZ_AUTOTUNE", 0), ("HZ_TC_CFG", cfg)):
        monkeypatch.setenv(k, str(v))
    rng = np.random.default_rng(sum(shape) + cfg)
    c = 1.5 + rng.random(shape)
    m, omega, npml, C = 1.0 / (c * c), W.omega_for_ppw(1.5, 9.0), 1, W.pml_constant(2.5)
    s = hz.Solver(m, omega, npml, C, 1, precision="mixed")
    s.factor()
    s.profile_begin(detail=True)
    solve_and_compare(s, shape, m, omega, npml, C, (17, 32, 33, 128), rng)
    s.profile_end()
    assert s.profile_kernel(1)["launches"] > 0
    s.close()


@pytest.mark.parametrize("shape,leaf", [((4, 5, 7), 1000), ((3, 4, 9), 8), ((9, 33, 10), 64), ((21, 24, 23), 256),
                                        ((12, 40, 44), 2000)])
def test_one_launch_substitution(shape, leaf, monkeypatch):
    """1 to 16 columns forced onto the one-launch kernel: one-node and one-tile trees, ragged tiles,
    split and whole reductions (the last box has nodes of over 8 half tiles)."""
    from paper_1801_08655_gb300 import build, hz
    build.build()
    monkeypatch.setenv("HZ_ONE_LAUNCH", "1")
    monkeypatch.setenv("HZ_LEAF", str(leaf))
    rng = np.random.default_rng(sum(shape))
    c = 1.5 + rng.random(shape)
    m, omega, npml, C = 1.0 / (c * c), W.omega_for_ppw(1.5, 9.0), 1, W.pml_constant(2.5)
    s = hz.Solver(m, omega, npml, C, 1, precision="mixed")
    s.factor()
    solve_and_compare(s, shape, m, omega, npml, C, (1, 2, 3, 8, 13, 16, 1), rng)
    s.close()


def test_one_launch_sparse_products_and_timeout(monkeypatch):
    """The trace operators' batches (skipped subtrees, several layers) agree with the per-phase launches;
    a wait that gives up is a status and leaves the counters usable for the next handle."""
    from paper_1801_08655_gb300 import build, hz
    build.build()
    p = W.small_problem(26, 4, 4, seed=5, R=3)
    out = {}
    for mode in ("0", "1"):
        monkeypatch.setenv("HZ_ONE_LAUNCH", mode)
        s = hz.Solver(p.m, p.omega, p.npml, p.C, p.n_layers, precision="mixed")
        s.factor()
        x = torch.randn(s.trace_shape(3), dtype=torch.complex128, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
        f = torch.from_numpy(p.rhs()).cuda()
        out[mode] = [s.apply_mpol(x), s.apply_precond(x), s.polarized_rhs(f), s.solve(f)[0]]
        s.close()
    for a, b in zip(out["0"], out["1"]):
        assert float((a - b).norm() / b.norm()) < 1e-5   # FP32 rounding, other summation orders
    monkeypatch.setenv("HZ_FACTOR_TC_MIN", "0")   # no bounded waits in the factorization
    ok = hz.Solver(p.m, p.omega, p.npml, p.C, p.n_layers, precision="mixed")
    ok.factor()
    monkeypatch.setenv("HZ_TC_WAIT_POLLS", "1")
    s = hz.Solver(p.m, p.omega, p.npml, p.C, p.n_layers, precision="mixed")
    s.factor()
    with pytest.raises(hz.HzError) as e:
        s.solve(f)
    assert e.value.status == hz.HZ_ERR_TIMEOUT
    u = ok.solve(f)[0]
    assert float((u - out["1"][3]).norm() / u.norm()) < 1e-5
    s.close()
    ok.close()
