"""Negative zeros are valid inputs (n_H >= 0, 0 <= x <= 1) and mean zero: a step, a batch, a server and the
allocation-free step on fields that hold them agree with the oracle, bookkeeping bit for bit, fields within
1e-12 (FP64) and 1e-5 (FP32) of the FP64 oracle."""
import ctypes as C

import numpy as np
import pytest

import oracle
from paper_2512_12466_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BOOK = ("rays", "splits", "escaped", "dropped_tau", "dropped_level", "segments", "secondary")


@pytest.fixture(scope="module")
def nyx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_12466_gb300 as m
    m.lib()
    return m


@pytest.fixture(scope="module")
def workload():
    w = I.random_small(17, 4, seed=77, x_mode="patchy", box_cm=17 * 2e22)
    rng = np.random.default_rng(78)
    w.n_h[rng.random(w.n_h.shape) < 0.2] = -0.0
    w.x_ion[rng.random(w.n_h.shape) < 0.2] = -0.0
    w.params["n_th_cm3"] = 0.3 * float(w.n_h.mean())
    return w


@pytest.fixture(scope="module")
def refs(workload):
    return [oracle.run_workload(workload, precision=p) for p in (0, 1)]


def dev(a, dtype=np.float64):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=dtype).ravel()).cuda()


def solver(nyx, w, precision):
    s = nyx.Solver(w.n, w.box_cm, precision=precision, **w.params)
    s.set_fields(dev(w.n_h), dev(w.x_ion))
    s.add_sources(dev(w.cells, np.int32), dev(w.ndot))
    return s


def check(refs, precision, g, st):
    for k in BOOK:
        assert list(st[k]) == list(refs[precision]["stats"][k]), k
    want = refs[0]["gamma"].ravel()
    assert np.linalg.norm(np.asarray(g).ravel() - want) / np.linalg.norm(want) < (1e-12 if precision == 0 else 1e-5)


@pytest.mark.parametrize("precision", [0, 1])
def test_step_batch_and_server(nyx, workload, refs, precision):
    w = workload
    s = solver(nyx, w, precision)
    g = torch.full((w.n ** 3,), np.nan, dtype=torch.float64, device="cuda")
    _, _, st = s.step(0.0, g, None)
    check(refs, precision, g.cpu().numpy(), st)
    ss = [solver(nyx, w, precision) for _ in range(2)]
    gs = [torch.full_like(g, np.nan) for _ in ss]
    b = nyx.Batch(ss)
    for g, st in zip(gs, b.run(gs, None)):
        check(refs, precision, g.cpu().numpy(), st)
    b.close()
    srv = nyx.Server(precision=precision)
    out = srv.poll(srv.submit(w.n, w.box_cm, w.n_h, w.x_ion, w.cells, w.ndot, **w.params), wait_s=60.0)
    check(refs, precision, out[0], out[2])
    srv.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_noalloc(nyx, workload, refs, precision):
    w = workload
    L = nyx.lib()
    L.rt_step_noalloc.argtypes = [C.POINTER(nyx.rt_config)] + [C.c_void_p] * 5 + [C.c_int64, C.c_void_p, C.c_void_p,
                                                                                C.POINTER(nyx.rt_stats), C.c_char_p, C.c_int32]
    cfg = nyx.rt_config_default(w.n, w.box_cm, precision=precision, **w.params)
    nh, x, cells, nd = dev(w.n_h), dev(w.x_ion), dev(w.cells, np.int32), dev(w.ndot)
    g = torch.full((w.n ** 3,), np.nan, dtype=torch.float64, device="cuda")
    st, err = nyx.rt_stats(), C.create_string_buffer(256)
    stream = torch.cuda.current_stream().cuda_stream
    rc = L.rt_step_noalloc(C.byref(cfg), stream, nh.data_ptr(), x.data_ptr(), cells.data_ptr(), nd.data_ptr(),
                           len(w.ndot), g.data_ptr(), None, C.byref(st), err, 256)
    assert rc == 0, err.value
    check(refs, precision, g.cpu().numpy(), nyx.stats_dict(st))
