"""The pivot-block kernel on boxes that are one tree node, so that every unknown goes through it: last blocks
of 1, 3, 11, 13, 16, 17, 21, 27, 31 and 32 unknowns, alone and behind full ones.  complex128: at most 225
unknowns, an unpivoted factorization of a well-conditioned operator, 1e-11; complex64: 4e-5."""
import numpy as np
import pytest
import scipy.sparse.linalg as spla

from oracle import discretization as D
from paper_1801_08655_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(3, 3, 3), (3, 3, 5), (3, 4, 4), (3, 3, 7), (4, 4, 4), (3, 5, 5), (3, 3, 9), (3, 3, 11),
                                   (3, 3, 13), (3, 5, 15)])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-11), ("mixed", 4e-5), ("mixed64", 5e-6)])
def test_one_node_boxes(shape, precision, tol, monkeypatch):
    from paper_1801_08655_gb300 import build, hz
    build.build()
    monkeypatch.setenv("HZ_LEAF", "1000")
    nz, ny, nx = shape
    rng = np.random.default_rng(nx * ny * nz)
    c = 1.5 + rng.random(shape)
    m, omega, npml, C = 1.0 / (c * c), W.omega_for_ppw(1.5, 9.0), 1, W.pml_constant(2.5)
    lu = spla.splu(D.assemble(m, omega, *[D.global_profiles(n, npml, C, omega) for n in (nx, ny, nz)]).tocsc())
    s = hz.Solver(m, omega, npml, C, 1, precision=precision)
    s.factor()
    for R in (1, 5):
        g = rng.standard_normal((R,) + shape) + 1j * rng.standard_normal((R,) + shape)
        ref = lu.solve(np.ascontiguousarray(g.reshape(R, -1).T)).T.reshape(g.shape)
        w = s.layer_solve(0, torch.from_numpy(g).cuda()).cpu().numpy()
        assert np.linalg.norm(w - ref) / np.linalg.norm(ref) < tol, (R, np.linalg.norm(w - ref) / np.linalg.norm(ref))
    s.close()
