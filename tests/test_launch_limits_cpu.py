"""Every launch finds its kernel's limit on dynamic shared memory raised on the device
it runs on, and no launch lowers a limit that another host thread's launch may
rely on: the launch code compiled against a pretended runtime of two devices
(launch_limits.cu; nothing runs on a GPU)."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_launch_limits(tmp_path):
    from paper_2307_02278_gb300 import build
    try:
        cc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    exe = str(tmp_path / "launch_limits")
    r = subprocess.run([cc, os.path.join(HERE, "launch_limits.cu"), "-o", exe, "-O1", "-std=c++17", build.ARCH, "-I",
                        build.INCLUDE, "-I", build.CSRC, "--expt-relaxed-constexpr"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
