"""The per-cell passes, the source stage and the chained levels at the sizes where their code paths change,
against the CPU oracle: grids around a pass's tile (1024 cells), catalogs around the one-block stage (2048
sources) and the sort's tile (1024 keys), bubble merging from shell tables and without them, opaque FP64
segments, and results by every way out. Bars as in test_gpu_parity: bookkeeping bit for bit, fields within
1e-12 (FP64) and 1e-5 (FP32) of the FP64 oracle."""
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


def dev(a, dtype):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=dtype).ravel()).cuda()


def rel(a, b):
    return float(np.linalg.norm(a.ravel() - b.ravel()) / max(np.linalg.norm(b), 1e-300))


def step(nyx, w, precision=0, **kw):
    s = nyx.Solver(w.n, w.box_cm, precision=precision, **kw)
    s.set_fields(dev(w.n_h, np.float64), dev(w.x_ion, np.float64))
    s.add_sources(dev(w.cells, np.int32), dev(w.ndot, np.float64))
    g = torch.full((w.n ** 3,), np.nan, dtype=torch.float64, device="cuda")
    h = torch.full_like(g, np.nan)
    _, _, st = s.step(0.0, g, h)
    return s, g.cpu().numpy(), h.cpu().numpy(), st


def check(nyx, w, precision=0, **kw):
    kw.setdefault("n_th_cm3", 0.01 * float(w.n_h.mean()))
    s, g, h, st = step(nyx, w, precision, **kw)
    ref = oracle.run_workload(w, precision=precision, **kw)
    ref64 = oracle.run_workload(w, precision=0, **kw)
    for k in BOOK:
        assert list(st[k]) == list(ref["stats"][k]), k
    assert (st["n_src_dedup"], st["n_src_emit"]) == (ref["stats"]["n_src_dedup"], ref["stats"]["n_src_emit"])
    bar = 1e-12 if precision == 0 else 1e-5
    assert rel(g, ref64["gamma"]) < bar and rel(h, ref64["heat"]) < bar
    return s, g, h, st


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n,x_mode", [(1, "mixed"), (10, "mixed"), (11, "neutral"), (16, "patchy"), (17, "thin")])
def test_field_pass_tiles(nyx, n, x_mode, precision):
    # 1, 1000, 1331, 4096 and 4913 cells: below a tile, just above one, whole tiles, a ragged last one
    w = I.random_small(n, 3, seed=500 + n, x_mode=x_mode, box_cm=n * 3e21)
    check(nyx, w, precision)[0].close()


def test_default_threshold_and_second_step(nyx):
    # the n_th default comes from the pass that copies the fields; a second step reuses it
    w = I.random_small(21, 4, seed=521, x_mode="patchy", box_cm=21 * 2e22)
    s, g, _, st = step(nyx, w)
    _, _, g2, st2 = s, None, *s.step(0.0)[::2]
    ref = oracle.run_workload(w, n_th_cm3=0.01 * float(w.n_h.mean()))
    assert rel(g, ref["gamma"]) < 1e-12 and rel(g2, ref["gamma"]) < 1e-12
    assert all(list(st[k]) == list(st2[k]) for k in BOOK)
    s.close()


@pytest.mark.parametrize("m", [1, 31, 33, 1024, 1025, 2047, 2048, 2049, 3100])
def test_catalog_sizes(nyx, m):
    # one block up to 2048 sources, tiles of 1024 keys above; a 12^3 grid of duplicates. The catalog is the
    # oracle's bit for bit: sorted cells, rates summed in input order
    w = I.random_small(12, m, seed=600 + m, x_mode="neutral", box_cm=12 * 3e21)
    s, _, _, st = check(nyx, w)
    cells, rates = w.cells.astype(np.int64), w.ndot
    key = (cells[:, 0] * 12 + cells[:, 1]) * 12 + cells[:, 2]
    order = np.argsort(key, kind="stable")
    want = {}
    for i in order:
        want[key[i]] = want[key[i]] + rates[i] if key[i] in want else rates[i]
    got_c, got_r = s.sources()
    got_c = np.asarray(got_c).reshape(-1, 3).astype(np.int64)
    assert list((got_c[:, 0] * 12 + got_c[:, 1]) * 12 + got_c[:, 2]) == list(want)
    assert np.array_equal(np.asarray(got_r), np.array(list(want.values())))
    s.close()


@pytest.mark.parametrize("dr,rmax,periodic", [(2.0, 16.0, 0), (1.5, 7.5, 1), (0.7, 5.0, 0), (2.0, 16.0, 1), (3.0, 2.0, 0)])
def test_bubble_radii(nyx, dr, rmax, periodic):
    # shells from the tables (dr a multiple of 2^-10, periodic grids wider than the shells), and the general
    # kernel (0.7; a periodic grid that the largest shells wrap around; no shell at all)
    w = I.random_small(30, 60, seed=700, x_mode="patchy", box_cm=30 * 2e22)
    x = w.x_ion.copy()
    x[4:19, 6:21, 3:18] = 1.0
    w.x_ion = x
    kw = dict(merge_mode=nyx.RT_MERGE_FORCED, merge_dr_cells=dr, merge_rmax_cells=rmax, merge_f_req=0.6, periodic=periodic)
    s, _, _, st = check(nyx, w, **kw)
    assert st["merged"] == 1
    s.close()


def test_sort_of_many_tiles(nyx):
    # more tiles than the sort has blocks (512 of 1024 keys): several tiles a block
    m = 600 * 1024 + 77
    rng = np.random.default_rng(31)
    w = I.random_small(64, 1, seed=950, x_mode="neutral", box_cm=64 * 3e21)
    cells, rates = rng.integers(0, 64, size=(m, 3)).astype(np.int32), rng.uniform(1, 2, m) * 1e48
    s = nyx.Solver(w.n, w.box_cm, n_th_cm3=1e-6)
    s.set_fields(dev(w.n_h, np.float64), dev(w.x_ion, np.float64))
    s.add_sources(dev(cells, np.int32), dev(rates, np.float64))
    s.step(0.0, torch.empty(w.n ** 3, dtype=torch.float64, device="cuda"), None)
    key = (cells[:, 0].astype(np.int64) * 64 + cells[:, 1]) * 64 + cells[:, 2]
    order = np.argsort(key, kind="stable")
    uniq, start = np.unique(key[order], return_index=True)
    got_c, got_r = s.sources()
    assert np.array_equal((got_c[:, 0].astype(np.int64) * 64 + got_c[:, 1]) * 64 + got_c[:, 2], uniq)
    for u in rng.integers(0, len(uniq), 2000):                   # sums in input order, bit for bit
        run = rates[order[start[u]: start[u + 1] if u + 1 < len(start) else m]]
        acc = run[0]
        for v in run[1:]:
            acc = acc + v
        assert got_r[u] == acc
    s.close()


@pytest.mark.parametrize("dx", [3e20, 2e21, 5e22, 7e23])
def test_opaque_segments_fp64(nyx, dx):
    # optical depths per segment from thin through the switch at 2 to far beyond (neutral gas)
    w = I.random_small(20, 6, seed=800, x_mode="neutral", mean_nh=1e-3, box_cm=20 * dx)
    check(nyx, w)[0].close()


def test_ways_out(nyx):
    # device buffers, overlapping device buffers (copied), host arrays and one result alone agree
    w = I.random_small(19, 5, seed=900, x_mode="patchy", box_cm=19 * 2e22)
    s, g, h, _ = step(nyx, w)
    n3 = w.n ** 3
    both = torch.zeros(n3 + 7, dtype=torch.float64, device="cuda")
    s.step(0.0, both[:n3], both[7:])
    assert rel(both[7:].cpu().numpy(), h) < 1e-14                # the later copy, heat, is whole
    gh, hh, _ = s.step(0.0)
    assert rel(np.asarray(gh), g) < 1e-14 and rel(np.asarray(hh), h) < 1e-14
    only = torch.zeros(n3, dtype=torch.float64, device="cuda")
    s.step(0.0, None, only)
    assert rel(only.cpu().numpy(), h) < 1e-14
    s.close()


@pytest.mark.parametrize("what", ["field", "source", "merge"])
def test_invalid_inputs_leave_results(nyx, what):
    # invalid device inputs are found while the step is enqueued: an error, and nothing written
    w = I.random_small(14, 5, seed=950, x_mode="patchy", box_cm=14 * 2e22)
    nh, cells = w.n_h.copy(), w.cells.copy()
    if what == "field":
        nh[3, 4, 5] = -1.0
    else:
        cells[2] = (0, 0, 99)
    s = nyx.Solver(w.n, w.box_cm, merge_mode=nyx.RT_MERGE_FORCED if what == "merge" else nyx.RT_MERGE_OFF)
    s.set_fields(dev(nh, np.float64), dev(w.x_ion, np.float64))
    s.add_sources(dev(cells, np.int32), dev(w.ndot, np.float64))
    g = torch.full((w.n ** 3,), 7.0, dtype=torch.float64, device="cuda")
    with pytest.raises(nyx.NyxError):
        s.step(0.0, g, None)
    assert bool((g == 7.0).all())
    s.set_fields(dev(w.n_h, np.float64), dev(w.x_ion, np.float64))
    s.clear_sources()
    s.add_sources(dev(w.cells, np.int32), dev(w.ndot, np.float64))
    s.step(0.0, g, None)
    assert bool((g != 7.0).all())
    s.close()


def test_batch_outputs(nyx):
    # a batch writes separate device buffers itself and copies overlapping ones; a solve without work in it
    ws = [I.random_small(n, k, seed=40 + n, x_mode="neutral", box_cm=n * 3e21) for n, k in ((9, 2), (16, 40), (23, 1))]
    ss = []
    for w in ws:
        s = nyx.Solver(w.n, w.box_cm)
        s.set_fields(dev(w.n_h, np.float64), dev(w.x_ion, np.float64))
        s.add_sources(dev(w.cells, np.int32), dev(w.ndot, np.float64))
        ss.append(s)
    b = nyx.Batch(ss)
    refs = [oracle.run_workload(w, n_th_cm3=0.01 * float(w.n_h.mean())) for w in ws]
    for _ in range(3):
        gs = [torch.full((w.n ** 3,), np.nan, dtype=torch.float64, device="cuda") for w in ws]
        hs = [torch.full((w.n ** 3,), np.nan, dtype=torch.float64, device="cuda") for w in ws]
        b.run(gs, hs)
        for g, h, r in zip(gs, hs, refs):
            assert rel(g.cpu().numpy(), r["gamma"]) < 1e-12 and rel(h.cpu().numpy(), r["heat"]) < 1e-12
        b.capture()
    one = torch.zeros(max(w.n for w in ws) ** 3, dtype=torch.float64, device="cuda")
    b.run([one[: w.n ** 3] for w in ws], None)                   # all three on one buffer: the last copy is whole
    assert rel(one.cpu().numpy(), refs[2]["gamma"]) < 1e-12
    b.close()
