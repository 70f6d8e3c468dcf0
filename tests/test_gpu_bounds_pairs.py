"""The node-pair kernels and the batched steps on the bounds-checked debug build
(libclbm_bc.so): no index outside its buffer (clbm_check and clbm_batch_check
would report CLBM_ERR_BOUNDS), and the bits of one node per thread or of single
lattices. Runs the cases of bounds_check_pairs.py in a child process."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_checked_build_finds_no_out_of_range_index_in_pairs():
    from paper_1801_04586_gb300.builder import build
    build(bounds_check=True)
    env = dict(os.environ, CLBM_LIBRARY="bounds_check")
    r = subprocess.run([sys.executable, os.path.join(HERE, "bounds_check_pairs.py")], env=env, capture_output=True,
                       text=True, timeout=1200)
    results = [json.loads(ln) for ln in r.stdout.splitlines() if ln.startswith("{")]
    bad = [x for x in results if not x["ok"]]
    assert not bad, bad
    assert r.returncode == 0, r.stderr[-2000:]
    assert len(results) == 21
