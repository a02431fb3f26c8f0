"""The launch code keeps nothing per process that belongs to a device: kernel attributes are set for the
current device whenever a batch or a factorization is prepared, and SM counts come from the handle's device.
A mutable function-local static would be such state, unguarded against other threads besides."""
import os
import re

from paper_1801_08655_gb300 import build


def test_no_mutable_function_local_statics():
    found = []
    for name in sorted(os.listdir(build.CSRC)):
        text = open(os.path.join(build.CSRC, name)).read()
        text = re.sub(r"/\*.*?\*/", "", re.sub(r"//[^\n]*", "", text), flags=re.S)
        for line in text.splitlines():
            if re.match(r"\s+static\s+(?!constexpr|const\b|inline|__)", line):
                found.append(f"{name}: {line.strip()}")
    assert not found, found


def test_every_large_shared_memory_launch_has_its_attribute_set():
    """Kernels launched with more than 48 KiB appear in a cudaFuncSetAttribute of the same file."""
    kernels = {"subst_tc.cu": ["k_subst_tc<", "k_subst_tcp<"], "subst_stream.cu": ["k_subst_stream<"],
               "factor_tc.cu": ["k_front_gemm<GEMM_L21>", "k_front_gemm<GEMM_SCHUR>", "k_front_gemm<GEMM_M21>"],
               "polarized.cu": ["k_trace_block2<8>", "k_trace_block2<16>"]}
    for name, ks in kernels.items():
        text = open(os.path.join(build.CSRC, name)).read()
        for k in ks:
            spots = [m.start() for m in re.finditer(re.escape(k), text)]
            assert any("MaxDynamicSharedMemorySize" in text[i:i + 250] for i in spots), (name, k)
