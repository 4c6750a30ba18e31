"""Batches on both sides of the planner's choices (transposed jobs, band-stream
jobs, inter-task chains of 8 to 24 rows and 4 to 32 lanes, query tracks): the
plan a batch gets by default against fixed ones, and against the CPU oracle on
a sample of the database.  Scores are int32; the bar is equality.
"""

import numpy as np
import pytest

import oracle
from workload import from_list, random_sequences, sample_indices
from workload.matrices import BLOSUM62

pytestmark = pytest.mark.gpu

QUERIES = {"one_residue": [1], "short": [60], "ordinary": [400], "two_bands": [1024], "long": [1301],
           "long_and_short": [2500, 60], "pair": [353, 471], "five": [100, 173, 300, 519, 900],
           "forty": list(range(20, 820, 20))}


@pytest.fixture(scope="module")
def api():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2412_08308_gb300 import api as _api
    from paper_2412_08308_gb300 import build

    build()
    oracle.build()
    return _api


def _scores(api, handle, queries, mode, **opts):
    batch = api.PreparedQueries(handle, queries.residues, queries.offsets, BLOSUM62, mode=mode,
                                opts=api.options(**opts) if opts else None)
    out = batch.search().cpu().numpy()
    batch.status()
    batch.close()
    return out


@pytest.mark.parametrize("n,long", [(1, 0), (30, 1), (700, 0), (3000, 2), (16384, 0), (16385, 1)])
@pytest.mark.parametrize("mode", ["packed", "int32"])
def test_default_plan(api, n, long, mode):
    source = random_sequences(500, 1, 3300, 0.0, 3300, 3300).as_list()[0]
    # `long` copies of a sequence past the intra-task cutover, a fragment of it in every query set
    seqs = random_sequences(501 + n, n, 300, 0.6, 1, 1000).as_list() + [source] * long
    db = from_list(seqs)
    handle = api.Database.from_sequences(db)
    idx = sample_indices(len(db), 40)
    for name, lengths in QUERIES.items():
        q = [random_sequences(600 + m, 1, m, 0.0, m, m).as_list()[0] for m in lengths]
        q[-1] = source[:lengths[-1]].copy()
        queries = from_list(q)
        got = _scores(api, handle, queries, mode)
        assert np.array_equal(got, _scores(api, handle, queries, mode, band_stream="never", rows_per_lane=12)), name
        if n <= 3000:
            assert np.array_equal(got, _scores(api, handle, queries, mode, band_stream="always")), name
        expected = oracle.scores(queries, db.subset(idx), BLOSUM62, 10, 2)
        assert np.array_equal(got[:, idx], expected), name
    handle.close()
