"""Databases with sequences past the intra-task cutover: one chain of the
intra-task kernel takes such a unit's columns one after the other, so short
queries belong to the transposed jobs however many other sequences there are.
The default plan must not hold inter- or intra-task work there, and its scores
must be those of the other kernels (integers: equal)."""

import numpy as np
import pytest

from workload import from_list, random_sequences
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


@pytest.mark.parametrize("n,long", [(0, [9000]), (300, [9000, 9000, 2048]), (12000, [9000] * 3), (16385, [9000]),
                                    (20000, [9000, 2100, 2048])])
@pytest.mark.parametrize("mode", ["packed", "int32"])
@pytest.mark.parametrize("q_len", [[60], [144], [400]])
def test_short_queries_leave_the_intra_task_kernel(api, n, long, mode, q_len):
    rng = np.random.Generator(np.random.PCG64(n + len(long)))
    seqs = random_sequences(n, n, 200, 0.4, 20, 900).as_list() if n else []
    db_s = from_list(seqs + [rng.integers(0, 20, size=k).astype(np.uint8) for k in long])
    qs = from_list([rng.integers(0, 20, size=k).astype(np.uint8) for k in q_len])
    db = api.Database.from_sequences(db_s)
    try:
        got = []
        for opts in (None, api.options(band_stream="never")):
            batch = api.PreparedQueries(db, qs.residues, qs.offsets, BLOSUM62, mode=mode, opts=opts)
            got.append(batch.search().cpu().numpy())
            batch.status()
            if opts is None:
                assert batch.info()[2] == 0, "inter- or intra-task work in the plan"
            batch.close()
    finally:
        db.close()
    assert np.array_equal(got[0], got[1])


# more than 16,384 peptides: up to 2,500,000 residues the transposed jobs are weighed too
@pytest.mark.parametrize("n,lo,hi", [(16384, 8, 30), (16385, 8, 30), (20000, 10, 60), (20000, 125, 125), (20001, 125, 125)])
@pytest.mark.parametrize("mode", ["packed", "int32"])
@pytest.mark.parametrize("q_len", [[255], [256], [1000], [30, 300]])
def test_peptide_databases(api, n, lo, hi, mode, q_len):
    rng = np.random.Generator(np.random.PCG64(n + hi))
    lens = rng.integers(lo, hi + 1, size=n)
    res = rng.integers(0, 20, size=int(lens.sum())).astype(np.uint8)
    qs = from_list([rng.integers(0, 20, size=k).astype(np.uint8) for k in q_len])
    db = api.Database(res, np.concatenate([[0], np.cumsum(lens)]))
    try:
        got = []
        for opts in (None, api.options(band_stream="never")):
            batch = api.PreparedQueries(db, qs.residues, qs.offsets, BLOSUM62, mode=mode, opts=opts)
            got.append(batch.search().cpu().numpy())
            batch.status()
            batch.close()
    finally:
        db.close()
    assert np.array_equal(got[0], got[1])


@pytest.mark.parametrize("band", ["auto", "always", "never"])
@pytest.mark.parametrize("mode", ["packed", "int32"])
def test_empty_database_and_empty_batch(api, band, mode):
    none = np.zeros(0, dtype=np.uint8)
    q = np.arange(20, dtype=np.uint8)
    for db_seqs, q_res, q_off in (([], q, [0, 20]), ([q, none], none, [0]), ([none, none], q, [0, 20]), ([], none, [0])):
        db = api.Database(np.concatenate([none] + db_seqs), np.cumsum([0] + [len(s) for s in db_seqs]))
        batch = api.PreparedQueries(db, q_res, np.array(q_off), BLOSUM62, mode=mode, opts=api.options(band_stream=band))
        out = batch.search()
        batch.status()
        assert out.shape == (len(q_off) - 1, len(db_seqs)) and int(out.sum()) == (
            0 if not any(len(s) for s in db_seqs) or len(q_off) == 1 else int(np.diag(BLOSUM62).sum()))
        batch.close()
        db.close()
