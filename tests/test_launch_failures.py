"""A launch that fails inside a call, with kernels of the same call on side
streams: before the call frees memory or returns, the handle's stream waits
for them. What the pattern scans of a row window are launched for, and what
happens without memory for them; the memory that learned sizing keeps; and that
side streams start after their memory is allocated.
CPU only: the object of api.cu is linked with a host stand-in for
the CUDA runtime and the kernels (host/fake_cuda.cpp)."""

import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_side_streams_are_waited_for_when_a_launch_fails(tmp_path):
    import paper_2206_07244_gb300 as ops
    from paper_2206_07244_gb300 import _buildlib
    ops.build()
    obj = os.path.join(_buildlib.BUILD, "api.cu.o")
    cuda = os.path.join(os.path.dirname(os.path.dirname(_buildlib._nvcc())) or "/usr/local/cuda", "include")
    exe = str(tmp_path / "fake_cuda")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", cuda, "-I", _buildlib.INCLUDE, "-I", _buildlib.CSRC,
                    os.path.join(HERE, "host", "fake_cuda.cpp"), obj, "-o", exe, "-lpthread", "-no-pie",
                    "-Wl,--unresolved-symbols=ignore-all"], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
