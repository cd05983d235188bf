"""A kernel's opt-in to more than 48 KB of shared memory, and the number of its CTAs that a device holds, belong to a
device.  The GEMMs' own object files are linked with a stand-in for the CUDA runtime (native/second_device.cpp) that has
two devices, and launched on both."""
import os
import subprocess

from conftest import ROOT

from paper_2310_04559_gb300 import build


def test_kernels_are_set_up_on_every_device(tmp_path):
    build.build()
    exe = str(tmp_path / "second_device")
    objs = [os.path.join(build.OUT_DIR, f) for f in ("gemm_crt.o", "gemm_tc.o")]
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc())))
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(cuda, "include"), "-I", os.path.join(ROOT, "include"),
                        os.path.join(ROOT, "tests", "native", "second_device.cpp"), *objs, "-o", exe, "-lpthread"],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
