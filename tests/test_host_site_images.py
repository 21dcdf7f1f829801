"""The images of X and Z that the compiler keeps per qubit through the gates and
records at every noise site (CPU, g++)."""
import os
import shutil
import subprocess

import pytest

from paper_2512_23037_gb300 import circuits as C

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.mark.parametrize("case", ["tiny6", "w42", "w97", "random40", "random90"])
def test_site_images_are_symplectic(tmp_path, case):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not available")
    if case.startswith("random"):  # every op kind, one and two key words
        circ, p = C.random_circuit(5, int(case[6:]), 500, t_frac=0.15, detectors=True, mpp_frac=0.1), 0.02
    else:
        circ, noise = C.workload(case)
        p = noise.p1
    out, ops = str(tmp_path / "check"), tmp_path / "ops.bin"
    csrc = os.path.join(ROOT, "paper_2512_23037_gb300", "csrc")
    subprocess.run([gxx, "-O1", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", "/usr/local/cuda/include",
                    os.path.join(HERE, "host", "site_image_check.cpp"), os.path.join(csrc, "compile.cpp"), "-o", out],
                   check=True, capture_output=True)
    ops.write_bytes(circ.array().tobytes())
    r = subprocess.run([out, str(ops), str(circ.n), repr(p)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.startswith("ok") and int(r.stdout.split()[1]) > 0, r.stdout + r.stderr
