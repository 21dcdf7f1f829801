"""The same call again: every shot's record and status byte.

Which lane or warp runs a shot, and when a warp hands its shots on, depends on
the order in which warps claim shots and on how many of them have ended, so it
changes from call to call. What a shot gives must not. Sizes at which evicted
shots go to the warp pass and at which they go to a second round and a wide
round, circuits of each lane size, one and two words a key.
"""
import numpy as np
import pytest

from paper_2512_23037_gb300 import circuits as C
from tests.test_gpu_parity import _random40

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


def _case(name):
    if name == "random40":
        return _random40(), C.Noise.uniform(5e-3)
    if name.startswith("win"):
        return C.windowed(12, n_data=32, n_anc=4, blocks=3, w=int(name[3:]), p=6e-3)
    return C.workload(name)[0], C.Noise.uniform({"w42": 2e-3, "w97": 1e-3}[name])


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("name,n", [("w42", 5000), ("w42", 300007), ("w42", (1 << 20) + 1), ("w97", 60001),
                                    ("random40", 100003), ("win5", 200003), ("win6", (1 << 20) + 1)])
def test_same_call_again(soft, name, n, precision):
    import torch
    S = soft
    circ, noise = _case(name)
    c = S.soft_compile_circuit(circ.array(), circ.n, noise, circ.cap)
    got = []
    for _ in range(4):
        rec = torch.zeros((n, c.info["record_words"]), dtype=torch.int64, device="cuda")
        status = torch.full((n,), 255, dtype=torch.uint8, device="cuda")
        r = S.soft_run_shots(c, n, 17, 5, precision=precision, record_mode=S.REC_ALL, d_records=rec.data_ptr(),
                             d_status=status.data_ptr())
        t = S.soft_tally(r)
        assert S.soft_run_diagnostics(r)[0] == 0
        r.free()
        assert [t[k] for k in KEYS[:4]] == [n] + [int((status == s).sum()) for s in (1, 2, 0)]
        got.append((rec, status, t))
    for rec, status, t in got[1:]:
        assert torch.equal(rec, got[0][0]) and torch.equal(status, got[0][1])
        assert [t[k] for k in KEYS] == [got[0][2][k] for k in KEYS]


@pytest.mark.parametrize("name,n,wide", [("w42", 300007, None), ("w42", (1 << 20) + 1, None),
                                         ("w42", (1 << 20) + 1, False), ("w97", 200003, None),
                                         ("random40", 100003, None), ("win5", (1 << 20) + 1, None)])
def test_every_shot_as_in_a_warp_of_its_own(soft, name, n, wide):
    """FP64: every record and status byte against the plain schedule, a warp per
    shot with sparse maps. Both round at 1e-15 and a shot samples some ten
    outcomes, so that one in 10^14 could differ: none may."""
    import torch
    S = soft
    circ, noise = _case(name)
    c = S.soft_compile_circuit(circ.array(), circ.n, noise, circ.cap)
    got = []
    for kw in ({"wide": wide}, {"lanes": False}):
        rec = torch.zeros((n, c.info["record_words"]), dtype=torch.int64, device="cuda")
        status = torch.full((n,), 255, dtype=torch.uint8, device="cuda")
        r = S.soft_run_shots(c, n, 40, 6, precision="fp64", record_mode=S.REC_ALL, d_records=rec.data_ptr(),
                             d_status=status.data_ptr(), **kw)
        S.soft_tally(r)
        r.free()
        got.append((rec, status))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("shots", [3000, 100000])
def test_same_batch_again(soft, shots, precision):
    """Lane sizes side by side, which race for the one list of the warp pass."""
    S = soft
    batch = [C.windowed(60 + k, n_data=28 + 2 * k, n_anc=4, blocks=3, w=w, p=4e-3) for k, w in enumerate((4, 5, 6, 3))]
    circs = [S.soft_compile_circuit(c.array(), c.n, nz, c.cap) for c, nz in batch]
    ns = [shots + 7 * k for k in range(len(batch))]
    got = []
    for _ in range(4):
        r = S.soft_run_batch(circs, ns, [0] * 4, 21, precision=precision)
        got.append([[S.soft_tally_batch(r, i)[k] for k in KEYS] for i in range(4)])
        r.free()
    assert np.array_equal(np.array(got), np.array([got[0]] * 4)) and [t[0] for t in got[0]] == ns


@pytest.mark.parametrize("name", ["w42", "w97", "random40", "win5"])
def test_entries_do_not_depend_on_the_schedule(soft, name):
    """FP32: the final map of every shot, bit for bit, whether evicted shots go on
    in a warp of their own (small runs) or in lanes again (with a wide round),
    in one chunk or several. (Sums over entries are FP64 and round to FP32
    alike but where one lies within 1e-16 of a tie.)"""
    S = soft
    circ, noise = _case(name)
    c = S.soft_compile_circuit(circ.array(), circ.n, noise, circ.cap)
    n, seen = 1500, []
    for kw in ({}, {"wide": True}, {"chunk_shots": 512}, {}):
        r = S.soft_run_shots(c, n, 3, 23, precision="fp32", record_mode=S.REC_ALL, capture_k=n, **kw)
        rec, status = S.soft_get_records(r, n)
        maps = []
        for i in range(n):
            signs, keys, vals = S.soft_get_state(r, i)
            order = np.lexsort((keys[:, 0], keys[:, 1]))
            maps.append((signs.tobytes(), keys[order].tobytes(), (vals[order] + 0.0).tobytes()))
        seen.append((rec, status, maps))
    for rec, status, maps in seen[1:]:
        assert np.array_equal(status, seen[0][1]) and np.array_equal(rec, seen[0][0])
        assert sum(a != b for a, b in zip(maps, seen[0][2])) == 0
