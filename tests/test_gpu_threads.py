"""Handles of different circuits on different threads and streams at once: the
launches of each take the shared memory of its own circuit (whose events and
records set it), whatever the others ask for meanwhile."""
import threading

import pytest

from paper_2512_23037_gb300 import circuits as C

pytestmark = pytest.mark.gpu
KEYS = ("shots", "discarded", "overflow", "kept", "logical_errors")


@pytest.fixture(scope="module")
def soft():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_23037_gb300 as S
    S.load()
    return S


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_circuits_of_different_length(soft, precision):
    import torch
    S = soft
    jobs = []
    for blocks in (2, 6, 14):
        circ, noise = C.windowed(12, n_data=32, n_anc=4, blocks=blocks, w=4, p=3e-3)
        jobs.append(S.soft_compile_circuit(circ.array(), circ.n, noise, circ.cap))

    def run(c, stream):
        r = S.soft_run_shots(c, 2000, 0, 9, precision=precision, stream=stream)
        t = S.soft_tally(r)
        r.free()
        return [t[k] for k in KEYS]

    want = [run(c, torch.cuda.current_stream()) for c in jobs]
    failed = []

    def work(k):
        try:
            stream = torch.cuda.Stream()
            for _ in range(150):
                got = run(jobs[k], stream)
                if got != want[k]:
                    failed.append((k, got, want[k]))
        except Exception as e:  # noqa: BLE001 (reported below, from the main thread)
            failed.append((k, repr(e)))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed[:3]
