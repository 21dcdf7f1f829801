"""The gradient's sums, to the last bits that cancelling leaves.

dF = (dN_fid - F dN_acc) / N_acc is the difference of two sweeps, and most
entries of a kept pattern's gradient are zero in theory: what is returned there
is what is left of the two sweeps' sums, some 1e-17 to 1e-12. The expected
values (tests/golden/gradient_two_sweeps.npz) are those of the plain form, every
error applied where it happens, two sweeps one after the other, each derivative
summed over a warp. The bar is that of equal arithmetic, relative 1e-9 (FP64) or
2e-5 (FP32), taken over the residues (below 1e-12) by themselves: sums in another
order, a fused product or a joined sweep are off by their whole size.
"""
import os

import numpy as np
import pytest

from paper_2512_23037_gb300 import circuits as C

pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "gradient_two_sweeps.npz")

# circuit, p, patterns, first, seed, precision: 42 qubits (errors carried past
# rotations and projections), small maps, maps above 32 entries (wide pass)
SETS = {
    "w42rz": ("w42rz", 1e-3, 3000, 7919, 1, "fp64"),
    "q3": (705, 2e-2, 200, 5, 5, "fp64"),
    "q3_fp32": (705, 2e-2, 200, 5, 5, "fp32"),
    "q4": (706, 8e-3, 2000, 6, 6, "fp64"),
    "q4_fp32": (706, 8e-3, 2000, 6, 6, "fp32"),
    "wide": (703, 2e-2, 400, 3, 3, "fp64"),
    "unobserved": ("unobserved", 3e-2, 400, 9, 9, "fp64"),
}


def unobserved():
    """No record is observed (F = 1), and no event is left for most errors to meet."""
    circ = C.Circuit(5, cap=256)
    rng = np.random.default_rng(11)
    for q in range(5):
        circ.gate(C.H, q)
    for k in range(30):
        circ.gate(C.RZ, int(rng.integers(5)), angle=0.0, param=k % 6, negate=bool(k % 3))
        a, b = (int(v) for v in rng.choice(5, size=2, replace=False))
        circ.gate(C.CX, a, b)
        circ.gate(int(rng.choice([C.H, C.S, C.T])), a)
    circ.detector([circ.measure(0)])
    for q in range(40):
        circ.gate(C.X, q % 5)
    return circ


def run_set(S, name):
    which, p, n, first, seed, precision = SETS[name]
    if which == "w42rz":
        circ, theta = C.workload(which)[0], C.rz_thetas(seed, 72)
    else:
        q = {705: 3, 706: 4, 703: 6}.get(which)
        circ = unobserved() if which == "unobserved" else C.random_param_circuit(which, q, 50 + 6 * q, 6)[0]
        theta = np.random.default_rng(seed if which == "unobserved" else which).uniform(-np.pi, np.pi, 6)
    c = S.soft_compile_circuit(circ.array(), circ.n, C.Noise.uniform(p), circ.cap)
    return [t.cpu().numpy() for t in S.soft_fidelity_grad(c, theta, n, first, seed, precision)]


@pytest.fixture(scope="module")
def soft():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_23037_gb300 as S
    S.load()
    return S


@pytest.mark.parametrize("name", list(SETS))
def test_sums_as_two_sweeps_leave_them(soft, name):
    with np.load(GOLDEN) as g:
        want = {k: g[f"{name}.{k}"] for k in ("status", "fid", "pacc", "row", "col", "val")}
    fid, pacc, grad, status = run_set(soft, name)
    assert np.array_equal(status, want["status"])
    bar = 1e-9 if SETS[name][5] == "fp64" else 2e-5
    ref = np.zeros_like(grad)
    ref[want["row"], want["col"]] = want["val"]
    tiny = np.abs(ref) < 1e-12
    assert np.count_nonzero(ref) > 100
    for part in (tiny, ~tiny):
        assert np.linalg.norm((grad - ref)[part]) <= bar * np.linalg.norm(ref[part])
    for got, key in ((fid, "fid"), (pacc, "pacc")):
        assert np.linalg.norm(got - want[key]) <= bar * np.linalg.norm(want[key])


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("sites", [255, 256, 257, 300])
def test_more_errors_than_a_pattern_may_have(soft, sites, precision):
    """An error at every site (p = 1 - 1e-12), none of which any event meets: a pattern of
    more than 256 errors is unsupported, one of 256 is not."""
    S = soft
    circ = C.Circuit(2, cap=4)
    circ.noiseless(True)
    circ.gate(C.RZ, 1, angle=0.3, param=0)
    circ.noiseless(False)
    for _ in range(sites):
        circ.gate(C.H, 0)
    c = S.soft_compile_circuit(circ.array(), circ.n, C.Noise.uniform(1.0 - 1e-12), circ.cap)
    assert c.info["n_sites"] == sites
    fid, pacc, grad, status = [t.cpu().numpy() for t in S.soft_fidelity_grad(c, [0.3], 40, 0, 1, precision)]
    assert np.all(status == (2 if sites > 256 else 0))
    assert np.all(fid == (0.0 if sites > 256 else 1.0)) and np.all(grad == 0.0)
