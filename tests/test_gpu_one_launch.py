"""The one-launch substitution (complex64 blocks of at most 16 columns) against the complex128 local
solves, one launch per substitution, at tolerances near its own error.

Tolerances: a local solve on complex64 factors is 1e-5 to 3e-5 off at 40^3 to 56^3 cells a layer, so 4e-5
on the boxes here (at most 20 000 cells); on rounded complex128 factors the products' FP32 rounding is
left, some 30 roundings of 6e-8 along a chain of products: 5e-6."""
import threading

import numpy as np
import pytest

from paper_1801_08655_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"mixed": 4e-5, "mixed64": 5e-6}


def one_layer(shape, precision, stream=None, seed=0):
    from paper_1801_08655_gb300 import hz
    rng = np.random.default_rng(seed + sum(shape))
    c = 1.5 + rng.random(shape)
    s = hz.Solver(1.0 / (c * c), W.omega_for_ppw(1.5, 9.0), 1, W.pml_constant(2.5), 1, precision=precision,
                  stream=stream)
    s.factor()
    return s


def sources(shape, R, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    return torch.randn((R,) + shape, dtype=torch.complex128, device="cuda", generator=g)


def rel(a, b):
    return float((a - b).norm() / b.norm())


@pytest.mark.parametrize("precision", ["mixed", "mixed64"])
@pytest.mark.parametrize("shape", [(9, 33, 10), (21, 24, 23), (24, 28, 30)])
def test_every_width_in_one_launch(shape, precision):
    from paper_1801_08655_gb300 import build
    build.build()
    s, ref = one_layer(shape, precision), one_layer(shape, "fp64")
    for R in range(1, 17):
        g = sources(shape, R, R)
        want = ref.layer_solve(0, g)
        s.layer_solve(0, g)
        s.profile_begin(detail=True)
        got = s.layer_solve(0, g)
        s.profile_end()
        assert s.profile_kernel(0)["launches"] == 1 and s.profile_kernel(1)["launches"] == 0, R
        assert rel(got, want) < TOL[precision], (R, rel(got, want))
    s.close()
    ref.close()


def test_agrees_with_the_launches_per_phase(monkeypatch):
    """Where the one launch is not taken (HZ_ONE_LAUNCH=0, or a device that cannot hold its whole grid), the
    launches per phase give the same solves, with more launches."""
    from paper_1801_08655_gb300 import build
    build.build()
    shape = (21, 24, 23)
    one = one_layer(shape, "mixed")
    monkeypatch.setenv("HZ_ONE_LAUNCH", "0")
    per_phase = one_layer(shape, "mixed")
    for R in (1, 4, 16):
        g = sources(shape, R, R)
        want = per_phase.layer_solve(0, g)
        per_phase.profile_begin(detail=True)
        per_phase.layer_solve(0, g)
        per_phase.profile_end()
        assert per_phase.profile_kernel(0)["launches"] > 4
        assert rel(one.layer_solve(0, g), want) < 5e-6   # the same factors, other summation orders
    one.close()
    per_phase.close()


def test_give_up_leaves_the_counters_usable(tmp_path):
    """On one handle: a wait that gives up is a status with a text that fits, the barrier counters are
    zero afterwards, and the next application is right."""
    import os
    import shutil
    import subprocess
    from paper_1801_08655_gb300 import build
    lib = build.build()
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "one_launch_give_up")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "native", "one_launch_give_up.cu")
    r = subprocess.run([nvcc, *build.ARCH, "-O2", "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC, src, "-o", exe,
                        "-L", os.path.dirname(lib), "-lhz", "-Xlinker", "-rpath=" + os.path.dirname(lib)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr


@pytest.mark.parametrize("precision", ["mixed", "mixed64"])
@pytest.mark.parametrize("forced", [True, False])
def test_wider_blocks_near_their_error(precision, forced, monkeypatch):
    """17 to 128 columns, on the tensor cores wherever that is allowed and as tuned: factors rounded from
    FP64 keep their digits at every width (the per-item kernel, or the CUDA cores up to 32 columns)."""
    from paper_1801_08655_gb300 import build
    build.build()
    if forced:
        for k, v in (("HZ_SUBST_TC", "1"), ("HZ_TC_MIN_TILES", "2"), ("HZ_AUTOTUNE", "0")):
            monkeypatch.setenv(k, v)
    shape = (21, 24, 23)
    s, ref = one_layer(shape, precision), one_layer(shape, "fp64")
    for R in (17, 24, 32, 33, 64, 100, 128):
        g = sources(shape, R, R)
        e = rel(s.layer_solve(0, g), ref.layer_solve(0, g))
        assert e < TOL[precision], (R, e)
    s.close()
    ref.close()


def test_two_handles_from_two_threads():
    """Handles on streams of their own, driven by a thread each: the cooperative launches of the two share
    the device, and every result is the one the handle gives alone."""
    from paper_1801_08655_gb300 import build
    build.build()
    shapes = [(21, 24, 23), (24, 28, 30)]
    hs = [one_layer(sh, "mixed", stream=torch.cuda.Stream()) for sh in shapes]
    widths = (1, 3, 8, 16)
    gs = [[sources(sh, R, R) for R in widths] for sh in shapes]
    torch.cuda.synchronize()
    alone = [[h.layer_solve(0, g) for g in row] for h, row in zip(hs, gs)]
    torch.cuda.synchronize()
    got = [[None] * len(widths) for _ in hs]
    failed = []

    def work(i):
        try:
            for _ in range(10):
                for k, g in enumerate(gs[i]):
                    got[i][k] = hs[i].layer_solve(0, g)
        except Exception as e:   # reported by the main thread
            failed.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed, failed
    for i in range(2):
        for a, b in zip(got[i], alone[i]):
            assert rel(a, b) < 5e-6
    for h in hs:
        h.close()
