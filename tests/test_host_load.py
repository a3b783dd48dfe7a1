"""A load that fails for lack of memory while one of its threads still reads the graph ends with the error code: the graph is given back
behind the thread.  In a process of its own, as memory read after it was given back ends one."""
import os
import subprocess
import sys

from tests.conftest import ROOT

LOAD = """
import numpy as np
from paper_2607_12324_b200 import build, emo
build.build()
n = 200_000      # (arrays of a size that the allocator maps and unmaps one by one)
rp, col = np.r_[0, np.arange(n)].astype(np.int64), np.arange(n - 1, dtype=np.int32)
lat, energy = np.ones((n, 2), np.int64), np.ones((n, 2))
for _ in range(3):
    try:
        emo.emo_graph_load(n, rp, col, None, 2, lat, energy, None, emo.EMO_F_HOST_ONLY | emo.EMO_F_GENERIC | emo.EMO_F_TEST_LONG_OOM)
    except emo.EmoError as e:
        assert e.code == -6, e
    else:
        raise AssertionError("the load did not fail")
print("refused")
"""


def test_failing_load_waits_for_its_threads():
    r = subprocess.run([sys.executable, "-c", LOAD], cwd=ROOT, capture_output=True, text=True, timeout=300, env=dict(os.environ))
    assert r.returncode == 0 and "refused" in r.stdout, (r.returncode, r.stderr)
