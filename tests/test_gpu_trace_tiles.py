"""Traceback over the edges of the walk's tiles, 144 steps x 16 lanes of 8 rows:
targets about 127 to 145 columns and multiples of the tile, query rows about
128 (16 lanes) and 256 (a band).  Every alignment must be the oracle's,
operation for operation (integer scores: no tolerance)."""

import numpy as np
import pytest

import oracle
from workload import from_list
from workload.matrices import BLOSUM62, DNA_SUBMAT

pytestmark = pytest.mark.gpu

M = [120, 127, 128, 129, 136, 144, 255, 256, 257, 383, 385, 640]
N = [112, 113, 127, 128, 129, 143, 144, 145, 160, 271, 287, 289, 433, 700]


@pytest.fixture(scope="module")
def api():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2412_08308_gb300 import api as _api
    from paper_2412_08308_gb300 import build

    build()
    oracle.build()
    return _api


@pytest.mark.parametrize("kind", ["identical", "ties", "long_gaps", "random"])
def test_tile_edges(api, kind):
    rng = np.random.Generator(np.random.PCG64(172))
    sm, go, ge = (BLOSUM62, 10, 2) if kind in ("identical", "random") else (DNA_SUBMAT, 1, 0)
    hi = 20 if sm is BLOSUM62 else 4
    base = rng.integers(0, hi, size=900).astype(np.uint8)
    if kind == "ties":  # one residue only: equal scores everywhere
        base[:] = 2

    def cut(n, target):
        if kind == "random":
            return rng.integers(0, hi, size=n).astype(np.uint8)
        if kind == "long_gaps":  # runs of E and of F longer than a tile is wide
            return np.delete(base, np.r_[60:100, 300:460] if target else np.r_[20:50, 150:240])[:n].copy()
        return base[:n].copy()

    qs, ts = from_list([cut(m, False) for m in M]), from_list([cut(n, True) for n in N])
    hits = [(i, j) for i in range(len(M)) for j in range(len(N))]
    db = api.Database.from_sequences(ts)
    try:
        got = api.traceback(db, qs.residues, qs.offsets, hits, sm, go, ge)
    finally:
        db.close()
    for (i, j), g in zip(hits, got):
        exp = oracle.align(qs[i], ts[j], sm, go, ge)
        assert g == exp, (kind, M[i], N[j], g[:5], exp[:5])
