"""GPU parity where the gap penalties choose the kernel: the penalties compiled
into a kernel (10 + 2k for proteins, 5 + 2k for DNA), their neighbours and the
extremes, in every kernel family, against the CPU oracle.  Scores are int32;
the bar is equality.
"""

import numpy as np
import pytest

import oracle
from workload import from_list, make_dna_pair, random_sequences
from workload.matrices import BLOSUM62, DNA_SUBMAT

pytestmark = pytest.mark.gpu

GAPS = [(10, 2), (10, 1), (9, 2), (11, 2), (5, 2), (0, 0), (0, 2), (12, 0), (1000, 12)]


@pytest.fixture(scope="module")
def api():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2412_08308_gb300 import api as _api
    from paper_2412_08308_gb300 import build

    build()
    oracle.build()
    return _api


@pytest.fixture(scope="module")
def protein_sets():
    # a query longer than two 512-row bands, one past a chunk of 24-row lanes,
    # short and single-residue ones; the longest query's copy scores past the rest
    q = random_sequences(71, 4, 120, 0.4, 1, 300).as_list()
    long = random_sequences(72, 1, 1100, 0.0, 1100, 1100).as_list()[0]
    q += [long, long[:769], long[:1]]
    db = random_sequences(73, 60, 200, 0.6, 1, 700).as_list() + [long[50:950]]
    return from_list(q), from_list(db)


@pytest.mark.parametrize("go,ge", GAPS)
@pytest.mark.parametrize("opts", [dict(band_stream="always"), dict(band_stream="always", band_rows=8),
                                  dict(band_stream="never", rows_per_lane=24),
                                  dict(band_stream="never", rows_per_lane=24, query_pairs=False),
                                  dict(band_stream="never", rows_per_lane=16, cutover=600),
                                  dict(band_stream="never", rows_per_lane=8, query_pairs=False),
                                  dict(band_stream="never", rows_per_lane=12)])
def test_penalties_in_every_kernel(api, protein_sets, go, ge, opts):
    queries, db = protein_sets
    expected = oracle.scores(queries, db, BLOSUM62, go, ge)
    handle = api.Database.from_sequences(db)
    for mode in ("packed", "int32"):
        batch = api.PreparedQueries(handle, queries.residues, queries.offsets, BLOSUM62, go, ge, mode,
                                    opts=api.options(**opts))
        got = batch.search().cpu().numpy()
        batch.status()
        batch.close()
        assert np.array_equal(got, expected), (mode, np.argwhere(got != expected)[:3])
    handle.close()


@pytest.mark.parametrize("go,ge", GAPS)
@pytest.mark.parametrize("rows", [0, 4, 8, 16, 24])
def test_pair_penalties(api, go, ge, rows):
    query, target = make_dna_pair(m=1500, n=1700, seed=74)
    got = api.align_pair(query, target, DNA_SUBMAT, go, ge, opts=api.pair_options(rows_per_lane=rows))
    assert got == oracle.score(query, target, DNA_SUBMAT, go, ge)
