"""Little free device memory: what runs with plenty of it still runs.

The rest of the memory is taken by one allocation, so that a call finds a given
number of bytes; its own allocations then fail in the ordinary way (an error
code), and it has to do with less.
"""
import contextlib

import numpy as np
import pytest

from paper_2512_23037_gb300 import circuits as C

pytestmark = pytest.mark.gpu
MB = 1 << 20


@pytest.fixture(scope="module")
def soft():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_23037_gb300 as S
    S.load()
    return S


@contextlib.contextmanager
def only(S, free):
    """All but `free` bytes of the device memory taken."""
    import torch
    S.soft_release_workspace()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    rest = torch.empty(torch.cuda.mem_get_info()[0] - free, dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        del rest
        torch.cuda.empty_cache()
        S.soft_release_workspace()


@pytest.mark.parametrize("wide", [None, True])
def test_run_in_smaller_chunks(soft, wide):
    """2^20 FP64 shots where their workspace does not fit: the same counts."""
    S = soft
    circ, noise = C.workload("w42")
    c = S.soft_compile_circuit(circ.array(), circ.n, noise, circ.cap)

    def run():
        r = S.soft_run_shots(c, 1 << 20, 0, 4, precision="fp64", wide=wide)
        t = S.soft_tally(r)
        r.free()
        return t

    want = run()
    with only(S, 100 * MB):
        assert run() == want


def test_compile_without_the_fate_tables(soft):
    """A circuit of 10^6 sites whose fate tables (64 MB a precision) find no memory:
    the same handle, the same records."""
    import torch
    S = soft
    circ = C.Circuit(8, cap=16)
    for k in range(250000):
        for q in range(4):
            circ.gate(C.H, (q + k) % 8)
    for q in range(8):
        circ.gate(C.T, q)
        circ.measure(q)
    ops, noise = circ.array(), C.Noise.uniform(1e-6)

    def records(c):
        r = S.soft_run_shots(c, 500, 0, 2, precision="fp64", record_mode=S.REC_ALL)
        rec, status = S.soft_get_records(r, 500)
        r.free()
        return rec, status

    before = torch.cuda.mem_get_info()[0]
    c = S.soft_compile_circuit(ops, circ.n, noise, circ.cap)
    took = before - torch.cuda.mem_get_info()[0]
    want = records(c)
    assert c.info["n_sites"] >= 1000000
    c.free()
    with only(S, took - 100 * MB):
        c = S.soft_compile_circuit(ops, circ.n, noise, circ.cap)
        got = records(c)
        c.free()
    assert all(np.array_equal(a, b) for a, b in zip(got, want))
