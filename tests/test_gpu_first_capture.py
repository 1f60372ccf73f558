"""pf_run_host's graph replay as the very first call of a process: everything its
routes query or load for the first time happens around the capture."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

SCRIPT = """
import numpy as np, sys
import oracle, synth
import paper_1910_03936_gb300 as pf
kind, dec, n, chunk, E = sys.argv[1], *map(int, sys.argv[2:])
if kind == "mixed":
    P = synth.generate(synth.SERVE, 5, n, kmax=60)
    P.E = np.minimum(P.E, E).astype(np.int16)
    args = dict(byte_off=P.read_off, E=P.E)
else:
    P = synth.generate(synth.SKEWED, 6, n, m=100, E=E, kmax=40)
    args = dict(length=100) if kind == "rows" else dict(byte_off=P.read_off)
c = pf.pf_create(0)
oa, oc = oracle.filter_batch(P)
rows = [0, 1] if dec == 3 else [dec - 1]
want = np.where(oa[rows[0]] == 1, oracle.verify_batch(P), P.E.astype(np.int32) + 1)
for _ in range(2):
    acc, cnt, dist = pf.pf_run_host(c, dec, P.reads, P.refs, E, chunk_pairs=chunk, **args)
    assert np.array_equal(acc, oa[rows]) and np.array_equal(cnt, oc[rows])
    assert np.array_equal(dist, want)
"""


@pytest.mark.parametrize("kind,dec,n,chunk,E", [
    ("mixed", 3, 40_500, 5_000, 25),        # one warp per pair
    ("mixed", 1, 400_500, 50_000, 25),      # grouped, 16 lanes
    ("ragged", 1, 480_100, 60_000, 13),     # 16 lanes and the list of long pairs
    ("ragged", 3, 4_800_100, 600_000, 10),  # the scheduler and the list
    ("rows", 2, 480_100, 60_000, 20),
])
def test_first_call(kind, dec, n, chunk, E):
    import os
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", SCRIPT, kind, str(dec), str(n), str(chunk), str(E)],
                       capture_output=True, text=True, timeout=300, cwd=root)
    assert r.returncode == 0, r.stderr[-2000:]
