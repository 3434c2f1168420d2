"""rt_set_fields recorded in a caller's CUDA graph: every replay brings new fields, so a step checks what is there
then (validity and the default threshold, from the mean density), whether the record is the library's kernel
(aligned device memory) or copies (misaligned memory), and whether it has been replayed at all."""
import numpy as np
import pytest

import oracle
from paper_2512_12466_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 16


@pytest.fixture(scope="module")
def nyx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_12466_gb300 as m
    m.lib()
    return m


def view(offset):
    """float64 storage at a byte offset of 0 or 4 modulo 8: (pointer, function that fills it)."""
    raw = torch.zeros(2 * N ** 3 + 2, dtype=torch.int32, device="cuda")
    words = raw[offset // 4: offset // 4 + 2 * N ** 3]

    def fill(a):
        words.copy_(torch.from_numpy(np.ascontiguousarray(a).ravel().view(np.int32)))
    return words.data_ptr(), fill


def record(nyx, s, stream, pn, px):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream, capture_error_mode="thread_local"):
        nyx.rt_set_fields(s.h, pn, px, nyx.RT_DEVICE)
    return g


@pytest.mark.parametrize("offset", [0, 4])
def test_replays_bring_new_fields(nyx, offset):
    ws = [I.random_small(N, 3, seed=60, x_mode="patchy", mean_nh=m, box_cm=N * 2e22) for m in (2e-4, 2e-2, 5e-5)]
    stream = torch.cuda.Stream()
    s = nyx.Solver(N, ws[0].box_cm, stream=stream.cuda_stream)
    (pn, fill_n), (px, fill_x) = view(offset), view(offset)
    fill_n(ws[0].n_h)
    fill_x(ws[0].x_ion)
    torch.cuda.synchronize()
    g = record(nyx, s, stream, pn, px)
    s.add_sources(ws[0].cells, ws[0].ndot)
    for w in ws:
        fill_n(w.n_h)
        fill_x(w.x_ion)
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            g.replay()
        gamma, _, st = s.step()
        ref = oracle.run_workload(w, n_th_cm3=0.01 * float(w.n_h.mean()))
        assert list(st["secondary"]) == list(ref["stats"]["secondary"])
        assert np.linalg.norm(gamma - ref["gamma"]) / np.linalg.norm(ref["gamma"]) < 1e-12
    bad = ws[0].n_h.copy()
    bad[1, 2, 3] = -1.0
    fill_n(bad)
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        g.replay()
    with pytest.raises(nyx.NyxError):
        s.step()
    torch.cuda.synchronize()
    s.close()


@pytest.mark.parametrize("offset", [0, 4])
def test_a_record_not_replayed_checks_nothing(nyx, offset):
    w = I.random_small(N, 3, seed=61, x_mode="patchy", box_cm=N * 2e22)
    stream = torch.cuda.Stream()
    s = nyx.Solver(N, w.box_cm, stream=stream.cuda_stream)
    bad = w.n_h.copy()
    bad[1, 2, 3] = -1.0
    s.set_fields(bad, w.x_ion)
    s.add_sources(w.cells, w.ndot)
    (pn, fill_n), (px, fill_x) = view(offset), view(offset)
    fill_n(w.n_h)
    fill_x(w.x_ion)
    torch.cuda.synchronize()
    g = record(nyx, s, stream, pn, px)
    with pytest.raises(nyx.NyxError):              # the fields in place are still the invalid ones
        s.step()
    with torch.cuda.stream(stream):
        g.replay()
    s.step()
    torch.cuda.synchronize()
    s.close()
