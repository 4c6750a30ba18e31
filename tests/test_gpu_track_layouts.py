"""The row-track lane tables a database keeps: however many heights, matrices,
modes and query lengths its searches went through, a plan that comes again
uploads no lane table.  Scores stay those of the other kernels (integers)."""

import numpy as np
import pytest

from workload import from_list
from workload.matrices import BLOSUM62

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2412_08308_gb300 import api as _api
    from paper_2412_08308_gb300 import build

    build()
    return _api


def test_layouts_stay_kept(api):
    rng = np.random.Generator(np.random.PCG64(31))
    seqs = [rng.integers(0, 20, size=int(L)).astype(np.uint8) for L in rng.integers(20, 900, size=600)]
    seqs += [rng.integers(0, 20, size=L).astype(np.uint8) for L in (1500, 4000)]
    db = api.Database.from_sequences(from_list(seqs))
    lanes = 8 * sum(len(s) // 24 for s in seqs)  # bytes: no lane table is smaller
    try:
        # (the largest score of a matrix sets which lengths take 16-bit tracks)
        for top in (11, 33, 36, 39, 42, 45, 48, 51, 54, 57, 60, 63):
            sm = BLOSUM62.copy()
            sm[17, 17] = top
            for mode in ("packed", "int32"):
                for m in (40, 1000):
                    q = rng.integers(0, 20, size=m).astype(np.uint8)
                    off = np.array([0, m])
                    got, h2d = [], []
                    for band in ("always", "always", "never"):
                        batch = api.PreparedQueries(db, q, off, sm, mode=mode, opts=api.options(band_stream=band))
                        got.append(batch.search().cpu().numpy())
                        batch.status()
                        h2d.append(batch.info()[0])
                        batch.close()
                    assert h2d[1] < lanes, (top, mode, m, h2d)
                    assert np.array_equal(got[0], got[2]) and np.array_equal(got[1], got[2])
    finally:
        db.close()
