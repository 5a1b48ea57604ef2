"""The bounds-checked build on the kernels of large lattices (four-step sweeps, ensemble
strips, D3Q19 sweeps) and on those that only a fixed launch runs alone: each is reached,
records no index fault, and has the one-step kernels' bits."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_large_lattice_kernels_record_no_index_fault():
    env = dict(os.environ, LBM_LIBRARY="checked")
    r = subprocess.run([sys.executable, os.path.join(HERE, "checked", "run_checked_large.py")], env=env,
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    out = json.loads(r.stdout.strip().splitlines()[-1])
    assert out["checked"] == 1 and out["max_diff"] == 0.0
    assert all(f == 0 for f in out["faults"]), out["faults"]
    assert all(n > 0 for n in out["reached"].values()), out["reached"]
    assert set(out["reached"]) == {"march", "march_kfield", "pairs", "nodes", "tiles", "sweep3", "strips", "general_single"}
