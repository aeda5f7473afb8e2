"""Index checks of the axis-separated step kernel: the LBF_DEBUG build checks its shared-memory and global indexes
against their buffers and reports a violation as LBF_EINTERNAL. Every form of it runs on shapes at the edges of its
tiles: lattice x storage x walls and force fields, both tiles, rows by TMA and by cp.async, two components, and the
clean rows of a split step (tests/debug_sweep_sep.py)."""
import os
import subprocess
import sys

import pytest

import debug_sweep_sep
from paper_2609_09160_gb300 import build

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_index_checked_axis_separated_kernel():
    lib = build.build(debug=True)
    env = dict(os.environ, LBF_LIBRARY=lib, PYTHONPATH=os.pathsep.join([os.path.dirname(HERE), HERE]))
    env.pop("LBF_KERNEL", None)
    res = subprocess.run([sys.executable, os.path.join(HERE, "debug_sweep_sep.py")], env=env, capture_output=True,
                         text=True, timeout=1500)
    failed = [l for l in res.stdout.splitlines() if "FAIL" in l]
    assert res.returncode == 0 and not failed, (failed[:10], res.stderr[-2000:])
    assert res.stdout.count(" ok") == len(list(debug_sweep_sep.cases()))
