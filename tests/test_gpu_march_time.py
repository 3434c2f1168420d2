"""rt_stats.ms_march is the time of the march launches, without the table builds and host waits that a
grid's first step has between them: the first step of a grid size reports about what the second does, far less
than its whole trace. (A build of this grid's FP64 tables takes tens of milliseconds, its march about one.)"""
import pytest

from paper_2512_12466_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_march_time_is_the_launches():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_12466_gb300 as nyx
    w = I.random_small(100, 4, seed=55, x_mode="thin", box_cm=100 * 7e20)
    s = nyx.Solver(w.n, w.box_cm, n_th_cm3=1e-6, n_min_ray=4.7)          # tables of its own
    s.set_fields(w.n_h.ravel(), w.x_ion.ravel())
    s.add_sources(w.cells.ravel(), w.ndot)
    first, second = s.step()[2], s.step()[2]
    third = s.step()[2]
    s.close()
    assert first["segments"] == second["segments"]
    assert 0.0 < first["ms_march"] < 0.5 * first["ms_trace"], first
    for st in (second, third):
        assert 0.0 < st["ms_march"] <= st["ms_trace"]
    # launches one by one on the first step, chained later: the spans differ by launch gaps and warm-up
    assert first["ms_march"] < 2.0 * min(second["ms_march"], third["ms_march"]) + 0.5, (first, second)
