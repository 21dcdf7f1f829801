"""The Pauli images that the compiler keeps per qubit through gates and
measurements, words and phases, against the decomposition over the tableau's
rows (CPU, g++)."""
import os
import shutil
import subprocess

import pytest

from paper_2512_23037_gb300 import circuits as C

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not available")
    out = str(tmp_path_factory.mktemp("host") / "image_phase_check")
    subprocess.run([gxx, "-O1", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", "/usr/local/cuda/include",
                    os.path.join(HERE, "host", "image_phase_check.cpp"), "-o", out], check=True, capture_output=True)
    return out


# one and two words a vector, one qubit short of and past the word's end; case B in most
@pytest.mark.parametrize("case", ["tiny6", "w42", "w97", "random3", "random40", "random63", "random64", "random65",
                                  "random90", "random128"])
def test_images_match_the_rows(checker, tmp_path, case):
    if case.startswith("random"):
        circ, p = C.random_circuit(5, int(case[6:]), 400, t_frac=0.15, detectors=True, mpp_frac=0.1), 0.02
    else:
        circ, noise = C.workload(case)
        p = noise.p1
    ops = tmp_path / "ops.bin"
    ops.write_bytes(circ.array().tobytes())
    r = subprocess.run([checker, str(ops), str(circ.n), repr(p)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.startswith("ok"), r.stdout + r.stderr
    sites, rotations, case_b = (int(v) for v in r.stdout.split()[1:])
    assert sites > 0 and rotations > 0 and (case_b > 0 or not case.startswith("random"))
