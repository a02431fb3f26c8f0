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
    prof = [D.global_profiles(n, npml, C, omega) for n in (nx, ny, nz)]
    A = D.assemble(m, omega, *prof).tocsc()
    for R in cols:
        g = rng.standard_normal((R,) + shape) + 1j * rng.standard_normal((R,) + shape)
        ref = spla.spsolve(A, g.reshape(R, -1).T).reshape(nz * ny * nx, R).T.reshape(g.shape)
        w = s.layer_solve(0, torch.from_numpy(g).cuda()).cpu().numpy()
        err = np.linalg.norm(w - ref) / np.linalg.norm(ref)
        assert err < 2e-4, (R, err)
    s.close()
