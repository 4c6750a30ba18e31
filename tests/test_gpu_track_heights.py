"""Transposed jobs at every size where their layout can go wrong: sequences at
the edges of lanes and bands of every height (8 to 24 rows, 256 to 768 rows per
band), longer ones whose bands run as a pipeline (with short sequences in the
lanes they leave free), batches of one and several queries, databases small
enough for one band and large enough for several per SM sub-partition.  Scores
are int32; the bar is equality with the CPU oracle.
"""

import numpy as np
import pytest

import oracle
from workload import from_list, random_sequences
from workload.matrices import BLOSUM62

pytestmark = pytest.mark.gpu

EDGES = [e + d for e in (8, 12, 16, 20, 24, 256, 384, 512, 640, 768, 1024) for d in (-1, 0, 1)] + [1, 1600, 2500]


@pytest.fixture(scope="module")
def api():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2412_08308_gb300 import api as _api
    from paper_2412_08308_gb300 import build

    build()
    oracle.build()
    return _api


def _edge_sequences(repeat):
    seqs = []
    for k, n in enumerate(EDGES * repeat):
        seqs += random_sequences(300 + k, 1, n, 0.0, n, n).as_list()
    return seqs


@pytest.mark.parametrize("mode", ["packed", "int32"])
@pytest.mark.parametrize("n_random,repeat", [(0, 1), (300, 2), (1000, 1), (1900, 3), (5200, 1)])
@pytest.mark.parametrize("lengths", [[144], [1], [17, 16, 15], [513, 60]])
def test_transposed_jobs(api, mode, n_random, repeat, lengths):
    seqs = _edge_sequences(repeat)
    if n_random:
        seqs += random_sequences(81, n_random, 300, 0.5, 20, 1000).as_list()
    db = from_list(seqs + [np.zeros(0, np.uint8)])
    queries = from_list([random_sequences(90 + m, 1, m, 0.0, m, m).as_list()[0] for m in lengths])
    handle = api.Database.from_sequences(db)
    batch = api.PreparedQueries(handle, queries.residues, queries.offsets, BLOSUM62, mode=mode,
                                opts=api.options(band_stream="always"))
    got = batch.search().cpu().numpy()
    batch.status()
    batch.close()
    handle.close()
    expected = oracle.scores(queries, db, BLOSUM62, 10, 2)
    assert np.array_equal(got, expected), np.argwhere(got != expected)[:3]
