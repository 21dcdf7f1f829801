"""The schedules a run may take (one-block and block-binned pre-pass, shots
finished there, evictions to the warp pass or to a second round, the affine and
the sparse warp maps, lane sizes side by side, the wide round) against the
oracle, and at sizes the oracle is too slow for against the plain schedule: a
warp per shot with sparse maps (lanes=False), which shares none of them.

Bars. Against the oracle: those of test_gpu_parity (equal but for shots with an
outcome within its band). Between two GPU schedules in one precision: FP32
rounding moves a probability by at most about 1e-6 (some ten roundings of
6e-8) and a shot samples about 5 outcomes that are not decided, so at most
1e-5 of the shots may differ; FP64 sums differ by their order only (1e-15), so
none do. A small constant covers the ones that do by chance.
"""
import numpy as np
import pytest

import oracle
from paper_2512_23037_gb300 import circuits as C
from tests.test_gpu_gradient import _compare as compare_gradients
from tests.test_gpu_parity import _random40, compare_records

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
    if name == "random40":  # every kind of event; few of its errors are decided early
        return _random40(), C.Noise.uniform(5e-3)
    if name.startswith("win"):  # win5: 32-entry lanes, win6: 64-entry lanes (FP32) or the affine warps
        return C.windowed(12, n_data=32, n_anc=4, blocks=3, w=int(name[3:]), p=6e-3)
    circ, _ = C.workload(name)
    return circ, C.Noise.uniform({"w42": 4e-3, "w97": 1.5e-3, "tiny6": 3e-2}[name])


def _allowed(n, precision):
    return 2 + (int(1e-5 * n) if precision == "fp32" else 0)


def _tallies_close(a, b, n, precision):
    assert a["shots"] == b["shots"] == n
    assert all(abs(a[k] - b[k]) <= _allowed(n, precision) for k in KEYS), (a, b)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("name", ["tiny6", "w42", "w97", "random40", "win5", "win6"])
def test_errors_carried_ahead(soft, precision, name):
    """Several errors per shot: carried alone or in pairs, meeting at one event,
    discarded in the pre-pass. Records and status of every shot."""
    S = soft
    circ, noise = _case(name)
    n = 1500
    c = S.soft_compile_circuit(circ.array(), circ.n, noise, circ.cap)
    r = S.soft_run_shots(c, n, 11, 29, precision=precision, record_mode=S.REC_ALL)
    rec, st = S.soft_get_records(r, n)
    assert S.soft_run_diagnostics(r)[0] == 0
    ref = oracle.run(circ, circ.n, noise, circ.cap, 29, 11, n, threads=8)
    assert compare_records(circ, noise, 29, 11, rec, st, ref, precision) <= 1 + n // 500
    tal = S.soft_tally(r)
    assert [tal[k] for k in KEYS[:4]] == [n] + [int(np.sum(st == s)) for s in (1, 2, 0)]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n", [1, 33, 8192, 8193])
@pytest.mark.parametrize("name", ["w42", "win5"])
def test_prepass_edges(soft, precision, name, n):
    """One shot, a ragged warp, the one-block pre-pass's last size and the next."""
    S = soft
    circ, noise = _case(name)
    c = S.soft_compile_circuit(circ.array(), circ.n, noise, circ.cap)
    runs = [S.soft_run_shots(c, n, 5, 3, precision=precision, record_mode=S.REC_ALL, lanes=lanes)
            for lanes in (True, False)]
    (ra, sa), (rb, sb) = (S.soft_get_records(r, n) for r in runs)
    assert np.sum((sa != sb) | np.any(ra != rb, axis=1)) <= (_allowed(n, precision) if n > 33 else 0)
    _tallies_close(S.soft_tally(runs[0]), S.soft_tally(runs[1]), n, precision)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("name,n,wide", [("w42", (1 << 20) + 1, None), ("w42", (1 << 20) + 1, False),
                                         ("win5", (1 << 20) + 1, None), ("win6", (1 << 20) + 1, None),
                                         ("w42", 1 << 22, None)])
def test_large_runs(soft, precision, name, n, wide):
    """Above the size at which evicted shots go to a second round, whose last
    warps list theirs, and a wide round follows, whose shots a warp resumes from
    their hand-over: the counts, and the first shots' records."""
    S = soft
    circ, noise = _case(name)
    c = S.soft_compile_circuit(circ.array(), circ.n, noise, circ.cap)
    k = 4096
    runs = [S.soft_run_shots(c, n, 0, 8, precision=precision, record_mode=S.REC_FIRST_K, record_k=k, lanes=lanes,
                             wide=wide) for lanes in (True, False)]
    (ra, sa), (rb, sb) = (S.soft_get_records(r, k) for r in runs)
    assert np.sum((sa != sb) | np.any(ra != rb, axis=1)) <= _allowed(k, precision)
    _tallies_close(S.soft_tally(runs[0]), S.soft_tally(runs[1]), n, precision)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("shots,graph", [(300, False), (40000, False), (40000, True), (400000, False)])
def test_batch_of_every_lane_size(soft, precision, shots, graph):
    """Circuits of 16-, 32- and 64-entry lanes in one batch, their launches side
    by side, with and without second rounds, and captured; against each
    circuit's own run."""
    import torch
    S = soft
    batch = [C.windowed(60 + k, n_data=28 + 2 * k, n_anc=4, blocks=3, w=w, p=4e-3) for k, w in enumerate((4, 5, 6, 3))]
    circs = [S.soft_compile_circuit(c.array(), c.n, nz, c.cap) for c, nz in batch]
    ns = [shots + 7 * k for k in range(len(batch))]
    firsts = [1000 * k for k in range(len(batch))]
    kw = {"stream": torch.cuda.Stream(), "graph": True, "chunk_shots": sum(ns) // 3} if graph else {}
    r = S.soft_run_batch(circs, ns, firsts, 21, precision=precision, **kw)
    for i, c in enumerate(circs):
        one = S.soft_run_shots(c, ns[i], firsts[i], 21, precision=precision, lanes=False)
        _tallies_close(S.soft_tally_batch(r, i), S.soft_tally(one), ns[i], precision)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("cap,first_cap", [(16, 0), (256, 0), (2048, 0), (2048, 64)])
def test_affine_maps_at_their_limits(soft, precision, cap, first_cap):
    """Maps that outgrow the lanes, the affine warps (1024 values in FP32, 256
    in FP64: the pass at the cap takes over) and the cap."""
    S = soft
    circ, noise = C.windowed(31, n_data=32, n_anc=4, blocks=4, w=6, p=1e-2)
    n = 1200
    c = S.soft_compile_circuit(circ.array(), circ.n, noise, cap)
    r = S.soft_run_shots(c, n, 0, 6, precision=precision, record_mode=S.REC_ALL, first_cap=first_cap)
    rec, st = S.soft_get_records(r, n)
    ref = oracle.run(circ, circ.n, noise, cap, 6, 0, n, threads=8)
    assert compare_records(circ, noise, 6, 0, rec, st, ref, precision) <= 1 + n // 500


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n_params,n_ops", [(1, 60), (2, 97), (31, 120)])
def test_gradient_terms_and_many_errors(soft, precision, n_params, n_ops):
    """Several errors per pattern, carried to the event that decides one of them;
    derivative terms summed 16 rotations at a time, of one parameter (each row
    the same), of two, and of more than there are rows."""
    circ, noise = C.random_param_circuit(810 + n_params, 5, n_ops, n_params=n_params, p=0.08)
    theta = np.random.default_rng(n_params).uniform(-np.pi, np.pi, n_params)
    _, status = compare_gradients(soft, circ, noise, theta, 40, 4, precision)
    assert not np.any(status == 2)
