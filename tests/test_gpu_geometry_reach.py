"""Geometry tables are built for the levels that rays reach and no others, although levels are launched one behind
the other before their counts are known, and rt_stats.table_levels names the levels whose rays read one: one
source in opaque gas, then a thin box of the same grid (all levels), then the opaque gas again with every table
in place. A child process reports the builds (NYXRT_GEOMETRY_TRACE)."""
import json
import os
import re
import subprocess
import sys

import numpy as np
import pytest

import oracle
from paper_2512_12466_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
N = 48

CHILD = r"""
import json, sys
import numpy as np
sys.path.insert(0, sys.argv[1])
import paper_2512_12466_gb300 as nyx
sys.path.insert(0, sys.argv[1] + "/tests")
from test_gpu_geometry_reach import workload
out = []
for kind in ("opaque", "thin", "opaque"):
    w = workload(kind)
    s = nyx.Solver(w.n, w.box_cm, stream=0, precision=int(sys.argv[2]), n_th_cm3=0.3 * float(w.n_h.mean()))
    s.set_fields(w.n_h.ravel(), w.x_ion.ravel())
    s.add_sources(w.cells.ravel(), w.ndot)
    sys.stderr.write("step " + kind + "\n")
    sys.stderr.flush()
    _, _, st = s.step()
    out.append({k: st[k] for k in ("rays", "segments", "secondary", "dropped_tau", "table_levels")})
    s.close()
print(json.dumps(out))
"""


def workload(kind):
    return I.random_small(N, 1, seed=41, x_mode="neutral" if kind == "opaque" else "thin",
                          box_cm=N * (2e23 if kind == "opaque" else 7e20))


@pytest.mark.parametrize("precision", [0, 1])
def test_tables_follow_the_rays(precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = subprocess.run([sys.executable, "-c", CHILD, ROOT, str(precision)], env=dict(os.environ, NYXRT_GEOMETRY_TRACE="1"),
                       capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stderr[-2000:]
    steps = json.loads(p.stdout.strip().splitlines()[-1])
    built = [set(int(m) for m in re.findall(r"entries level (\d+) .*: built", part)) for part in p.stderr.split("step ")[1:]]
    reached = [{l for l, r in enumerate(st["rays"]) if r} for st in steps]
    assert len(reached[0]) < len(reached[1]) - 2, reached           # the opaque step ends levels earlier
    assert built == [reached[0], reached[1] - reached[0], set()]
    for st, levels in zip(steps, reached):
        assert st["table_levels"] == sum(1 << l for l in levels)
    assert steps[0] == steps[2]
    for st, kind in zip(steps, ("opaque", "thin")):
        w = workload(kind)
        ref = oracle.run_workload(w, precision=precision, n_th_cm3=0.3 * float(w.n_h.mean()))["stats"]
        for k in ("rays", "segments", "secondary", "dropped_tau"):
            assert list(st[k]) == list(ref[k]), k


@pytest.mark.parametrize("where", ["host", "device"])
def test_chemistry_on_a_grid_without_tables(where):
    # the update and the results enqueued behind a trace that stops before an unbuilt level wait for its rays
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_12466_gb300 as nyx
    w = I.stromgren_test("A", 32)
    kw = {k: w.params[k] for k in ("tau_max", "chem_iterate", "alpha_B", "clumping", "C_H")}
    kw.update(n_th_cm3=1e-5, n_min_ray=4.3 if where == "host" else 4.4)
    dt = 10.0 * I.MYR_S
    ref = oracle.run(w.n_h, w.x_ion, w.cells, w.ndot, w.box_cm, dt_s=dt, **kw)
    out = torch.full((2, w.n ** 3), np.nan, dtype=torch.float64, device="cuda")
    for _ in range(2):                                      # without tables, then with
        s = nyx.Solver(w.n, w.box_cm, **kw)
        s.set_fields(w.n_h.ravel(), w.x_ion.ravel())
        s.add_sources(w.cells.ravel(), w.ndot)
        gamma, heat, st = s.step(dt) if where == "host" else s.step(dt, out[0], out[1])
        gamma, heat, x = [np.asarray(a.cpu() if hasattr(a, "cpu") else a).ravel() for a in (gamma, heat, s.get_x())]
        s.close()
        assert sum(1 for r in st["rays"] if r) > 4
        assert abs(st["chem_iters"] - ref["stats"]["chem_iters"]) <= 1
        for got, want in ((gamma, ref["gamma"]), (heat, ref["heat"]), (x, ref["x"])):
            assert np.linalg.norm(got - want.ravel()) / np.linalg.norm(want) < 1e-8
