"""The vetter's kernels get their shared-memory limits on every device that a vetter is made on."""
import ctypes
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_limits_on_every_device(tmp_path):
    from paper_2509_26279_gb300 import _build
    _build.build()
    so = str(tmp_path / "vet.so")
    subprocess.run([_build._nvcc(), *_build.ARCH, *_build.NVCC_FLAGS, "-shared", "-o", so,
                    os.path.join(ROOT, "tests", "native", "vet_devices.cu"), _build.LIB, "-Xlinker",
                    "-rpath=" + _build.OUT_DIR], check=True)
    lib = ctypes.CDLL(so)
    first, second = lib.limits_after_create(0), lib.limits_after_create(1)
    assert first > 0 and second == first
