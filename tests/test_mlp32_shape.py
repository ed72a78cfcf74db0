"""The persistent grid of the FP32 travel-time kernel is resident at once: an SM
holds the CTAs per SM of every width and form (228 KB of shared memory, 1 KB a CTA
reserved, 64 warps, 65,536 registers at 128 a thread).  On the CPU, from the header
the kernel uses."""
import ctypes as C
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2508_12117_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("mlp32") / "mlp32_harness.so")
    subprocess.run(["g++", "-O2", "-fPIC", "-shared", "-std=c++17", "-I", CSRC,
                    os.path.join(ROOT, "tests", "host", "mlp32_harness.cpp"), "-o", so], check=True, capture_output=True)
    return C.CDLL(so)


@pytest.mark.parametrize("wide", [0, 1])
@pytest.mark.parametrize("H", [32, 64, 128, 256])
def test_grid_is_resident_at_once(lib, H, wide):
    out = (C.c_longlong * 4)()
    assert lib.mlp32_shape(H, wide, out) == 0
    ctas, threads, smem, tile = out
    assert tile == (64 if wide else 32)
    assert ctas * (smem + 1024) <= 228 * 1024
    assert ctas * threads <= 2048
    assert not wide or ctas * threads * 128 <= 65536
