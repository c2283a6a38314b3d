"""The bench's reference arm, on CPU: its pair list is the oracle's, its sample and
overlap counts are those of the library's planner, and it loads nothing of the
library."""
import os
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402
from ofm_inputs import make_workload  # noqa: E402
from oracle import ofm_oracle as O  # noqa: E402


@pytest.mark.parametrize("name", ["tiny", "alkane", "polymer", "lattice4"])
def test_sample_of_the_oracles_pairs(name):
    wl = make_workload(name)
    assert bench._pair_list(wl.grid, wl.frags) == O.pair_list(wl.grid, wl.frags)
    from paper_1011_4764_gb300 import build, ofm
    build.build()
    pairs, cnt, _ = ofm.plan_pairs(wl.grid, wl.frags)
    pick = np.sort(np.random.default_rng(0).choice(len(pairs), size=min(8, len(pairs)), replace=False))
    got, shared = bench._sample_pairs(wl, 8)
    assert got == [pairs[i] for i in pick]
    assert [tuple(map(int, s)) for s in shared] == [tuple(map(int, cnt[i])) for i in pick]


def test_reference_arm_loads_no_library():
    code = ("import sys, bench; bench.run_reference(type('A', (), dict(workload='tiny', warmup=0, steps=1, gpus=1))());"
            "assert not [m for m in sys.modules if 'gb300' in m];"
            "assert 'libofm' not in open('/proc/self/maps').read()")
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert '"impl": "reference"' in r.stdout
