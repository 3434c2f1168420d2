"""Levels launched before their counts are known take ray buffers for every ray they might hold. Where such a
buffer cannot be had the step goes on with the rays there are: with the tables in place, a second solver's step
whose k-th allocation fails (NYXRT_FAULT_ALLOC, on the host) returns RT_ENOMEM only for the first, level 0's own,
and equals the oracle either way. Each case runs in a child process."""
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

CHILD = r"""
import json, sys
import numpy as np
sys.path.insert(0, sys.argv[1])
import paper_2512_12466_gb300 as nyx
from paper_2512_12466_gb300 import inputs as I
w = I.random_small(24, 2, seed=9, x_mode="thin", box_cm=24 * 7e20)
for turn in ("first", "second"):
    s = nyx.Solver(w.n, w.box_cm, stream=0, n_th_cm3=1e-6)
    s.set_fields(w.n_h.ravel(), w.x_ion.ravel())
    s.add_sources(w.cells.ravel(), w.ndot)
    sys.stderr.write("step " + turn + "\n")
    sys.stderr.flush()
    failed = 0
    try:
        g, _, st = s.step()
    except nyx.NyxError as e:
        failed = e.code
        g, _, st = s.step()
    sys.stderr.write("step done\n")
    sys.stderr.flush()
    s.close()
np.save(sys.argv[2], g)
print(json.dumps({"failed": failed, "rays": st["rays"]}))
"""


def run_child(tmp_path, env_extra):
    out = tmp_path / "gamma.npy"
    p = subprocess.run([sys.executable, "-c", CHILD, ROOT, str(out)], env=dict(os.environ, **env_extra), capture_output=True,
                       text=True, timeout=300)
    assert p.returncode == 0, p.stderr[-2000:]
    return json.loads(p.stdout.strip().splitlines()[-1]), np.load(out), p.stderr


def test_a_step_needs_memory_only_for_its_rays(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    w = I.random_small(24, 2, seed=9, x_mode="thin", box_cm=24 * 7e20)
    ref = oracle.run_workload(w, n_th_cm3=1e-6)
    _, _, err = run_child(tmp_path, {"NYXRT_FAULT_ALLOC_TRACE": "1"})
    part = err[err.index("step second"):]
    ords = [int(k) for k in re.findall(r"nyxrt-dalloc (\d+)", part[:part.index("step done")])]
    assert len(ords) >= 3, err
    for k in (ords[0], ords[1], ords[-1]):
        res, g, _ = run_child(tmp_path, {"NYXRT_FAULT_ALLOC": str(k)})
        assert res["failed"] == (-2 if k == ords[0] else 0), (k, ords, res)
        assert res["rays"] == ref["stats"]["rays"]
        assert np.linalg.norm(g - ref["gamma"]) / np.linalg.norm(ref["gamma"]) < 1e-12
