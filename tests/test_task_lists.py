"""Work lists of the substitution (CUDA-core tasks, tensor-core items, one-launch tasks, rows to clear) and of
the factorization's tensor-core products, walked on the host with the kernels' own index arithmetic:
every tile, row and update index in range, every product covered exactly once, dependent phases in order."""
import os
import shutil
import subprocess

import pytest

from paper_1801_08655_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def walker(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    lib = build.build()
    exe = str(tmp_path_factory.mktemp("native") / "substitution_lists")
    r = subprocess.run([nvcc, *build.ARCH, "-O2", "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC,
                        os.path.join(HERE, "native", "substitution_lists.cu"), "-o", exe, "-L", os.path.dirname(lib), "-lhz",
                        "-Xlinker", "-rpath=" + os.path.dirname(lib)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


# nx, ny, nz, npml, layers, leaf: one node; nodes of a few cells; ragged boxes with slabs of two thicknesses; the
# default leaf; flat and long boxes
@pytest.mark.parametrize("box", [(7, 5, 4, 0, 1, 1000), (9, 4, 3, 0, 1, 8), (10, 33, 9, 1, 1, 64), (23, 24, 21, 3, 3, 256),
                                 (67, 51, 59, 8, 5, 256), (13, 17, 61, 5, 7, 64), (70, 11, 30, 4, 2, 256)])
def test_every_task_stays_in_its_arrays(walker, box):
    r = subprocess.run([walker, *map(str, box)], capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout + r.stderr
    assert " tasks, " in r.stdout
