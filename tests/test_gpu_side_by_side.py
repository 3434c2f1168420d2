"""Launches that start in the tail of the one before (levels chained on a stream) beside another solver's work, and
a batch whose light solves pass from one launch to the next (2^22 measured segments a launch): results equal to the
oracle and to single steps."""
import threading

import numpy as np
import pytest

import oracle
from paper_2512_12466_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BOOK = ("rays", "splits", "escaped", "dropped_tau", "dropped_level", "segments", "secondary", "visit_hash")


@pytest.fixture(scope="module")
def nyx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_12466_gb300 as m
    m.lib()
    return m


def solver(nyx, w, precision, stream):
    s = nyx.Solver(w.n, w.box_cm, stream=stream, precision=precision, n_th_cm3=0.3 * float(w.n_h.mean()),
                   flags=nyx.RT_FLAG_VISIT_HASH)
    s.set_fields(w.n_h.ravel(), w.x_ion.ravel())
    s.add_sources(w.cells.ravel(), w.ndot)
    return s


@pytest.mark.parametrize("precision", [0, 1])
def test_two_solvers_on_two_streams(nyx, precision):
    ws = [I.random_small(20 + 9 * k, 3, seed=30 + k, x_mode=("thin", "patchy")[k], box_cm=(20 + 9 * k) * 2e21) for k in range(2)]
    refs = [oracle.run_workload(w, precision=precision, n_th_cm3=0.3 * float(w.n_h.mean())) for w in ws]
    wrong = []

    def work(k):
        stream = torch.cuda.Stream()
        s = solver(nyx, ws[k], precision, stream.cuda_stream)
        for turn in range(25):
            gamma, _, st = s.step()
            want = refs[k]["gamma"]
            if any(list(np.atleast_1d(st[q])) != list(np.atleast_1d(refs[k]["stats"][q])) for q in BOOK) or \
                    np.linalg.norm(gamma - want) / np.linalg.norm(want) > (1e-12 if precision == 0 else 1e-5):
                wrong.append((k, turn))
        s.close()

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong


@pytest.mark.parametrize("precision", [0, 1])
def test_light_solves_across_launches(nyx, precision):
    # measured segments on both sides of the launch's 2^22, group_bytes too small for any two solves
    ws = [I.random_small(n, k, seed=70 + n, x_mode="thin", box_cm=n * 7e20) for n, k in ((40, 1), (40, 3), (12, 2), (48, 1), (44, 2))]
    stream = torch.cuda.current_stream().cuda_stream
    ss = [solver(nyx, w, precision, stream) for w in ws]
    ref = [s.step() for s in ss]
    segments = [sum(st["segments"]) for _, _, st in ref]
    assert max(segments) < 2 ** 22 < sum(segments)
    b = nyx.Batch(ss)
    b.set_params(group_bytes=1 << 20)
    for turn in range(3):                                   # without measured work, with it, replayed
        gs = [np.empty((w.n,) * 3) for w in ws]
        for g, st, (want, _, want_st) in zip(gs, b.run(gs, None), ref):
            assert all(st[q] == want_st[q] for q in BOOK)
            assert np.linalg.norm(g - want) / np.linalg.norm(want) < (1e-12 if precision == 0 else 1e-10)
        if turn == 1:
            b.capture()
    b.close()
