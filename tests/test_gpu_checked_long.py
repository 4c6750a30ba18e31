"""The checked build (-DSW_CHECK) on long pairs and tracebacks: rings that wrap,
several bands and rounds of bands, empty and one-residue hits.  Each case runs
in a process bound to libswgb_check.so and must match the CPU oracle with no
index reported (sw_align_pair and sw_traceback fail on one)."""

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r'''
import sys
import numpy as np
sys.path.insert(0, ROOT)
from paper_2412_08308_gb300 import build
import paper_2412_08308_gb300._native as N
N.use_library(build(checked=True))
from paper_2412_08308_gb300 import api
import oracle
from workload import from_list, make_dna_pair
from workload.matrices import BLOSUM62, DNA_SUBMAT
oracle.build()

for m, n in ((1, 1), (129, 17), (1500, 1700), (3000, 513), (700, 3000)):
    q, t = make_dna_pair(m=m, n=n, seed=m + n)
    exp = oracle.score(q, t, DNA_SUBMAT, 5, 2)
    for rows in (0, 4, 8, 16, 24):
        for opts in (dict(), dict(ring_columns=256, max_ctas=1), dict(ring_columns=256, band_warps=1, max_ctas=2)):
            got = api.align_pair(q, t, DNA_SUBMAT, 5, 2, opts=api.pair_options(rows_per_lane=rows, **opts))
            assert got == exp, ("pair", m, n, rows, opts, got, exp)

rng = np.random.Generator(np.random.PCG64(19))
M, T = [0, 1, 8, 255, 256, 257, 700], [0, 1, 16, 17, 300, 513]
qs = from_list([rng.integers(0, 20, size=m).astype(np.uint8) for m in M])
ts = [rng.integers(0, 20, size=n).astype(np.uint8) for n in T]
ts[4][:] = qs[6][100:400]
ts = from_list(ts)
hits = [(i, j) for i in range(len(M)) for j in range(len(T))]
db = api.Database.from_sequences(ts)
got = api.traceback(db, qs.residues, qs.offsets, hits, BLOSUM62)
db.close()
for (i, j), g in zip(hits, got):
    assert g == oracle.align(qs[i], ts[j], BLOSUM62, 10, 2), ("trace", M[i], T[j])
print("checked build: all cases exact, no index reported")
'''


def test_checked_pairs_and_tracebacks():
    r = subprocess.run([sys.executable, "-c", SCRIPT.replace("ROOT", repr(ROOT), 1)], capture_output=True, text=True,
                       timeout=1800, cwd=ROOT)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    assert "no index reported" in r.stdout
