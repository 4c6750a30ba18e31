"""Traceback over the edges of its tiling: bands of 32 lanes x 8 rows, blocks
of 16 columns, walk tiles of 64 steps x 8 lanes.  Every alignment must be the
oracle's, operation for operation (integer scores: no tolerance)."""

import numpy as np
import pytest

import oracle
from workload import from_list
from workload.matrices import BLOSUM62, DNA_SUBMAT

pytestmark = pytest.mark.gpu

M = [1, 7, 8, 9, 63, 64, 65, 255, 256, 257, 511, 513, 1025]
N = [1, 15, 16, 17, 63, 65, 300, 1100]


@pytest.fixture(scope="module")
def api():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2412_08308_gb300 import api as _api
    from paper_2412_08308_gb300 import build

    build()
    oracle.build()
    return _api


@pytest.mark.parametrize("kind", ["identical", "ties", "gapped", "random"])
def test_band_and_tile_edges(api, kind):
    rng = np.random.Generator(np.random.PCG64(171))
    sm, go, ge = (BLOSUM62, 10, 2) if kind in ("identical", "random") else (DNA_SUBMAT, 1, 1)
    hi = 20 if sm is BLOSUM62 else 4
    base = rng.integers(0, hi, size=1200).astype(np.uint8)
    if kind == "ties":  # one residue only: equal scores everywhere
        base[:] = 1

    def cut(n, step):
        if kind == "random":
            return rng.integers(0, hi, size=n).astype(np.uint8)
        if kind == "gapped" and step:  # every 37th residue left out: long alignments with many gaps
            return np.delete(base, np.arange(5, len(base), 37))[:n]
        return base[:n].copy()

    qs, ts = from_list([cut(m, 0) for m in M]), from_list([cut(n, 1) for n in N])
    hits = [(i, j) for i in range(len(M)) for j in range(len(N))]
    db = api.Database.from_sequences(ts)
    try:
        got = api.traceback(db, qs.residues, qs.offsets, hits, sm, go, ge)
    finally:
        db.close()
    for (i, j), g in zip(hits, got):
        exp = oracle.align(qs[i], ts[j], sm, go, ge)
        assert g == exp, (kind, M[i], N[j], g[:5], exp[:5])
