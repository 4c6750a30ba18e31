"""Batches of many query lengths against a small database: planning them must not
cost many times what it costs where nothing is left to choose (the lanes per
chain given), and every floor of lanes, rows per lane and mode that the planner
weighs keeps the oracle's scores."""

import time

import numpy as np
import pytest

import oracle
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


def _batch(lens, n, hi):
    rng = np.random.Generator(np.random.PCG64(n + len(lens)))
    db = from_list([rng.integers(0, 20, size=int(k)).astype(np.uint8) for k in rng.integers(1, hi, size=n)])
    return db, from_list([rng.integers(0, 20, size=int(k)).astype(np.uint8) for k in lens])


# 30 floors x rows planned in full took 6 to 7 times the planning with the lanes given
def test_planning_time_of_many_lengths(api):
    db_s, qs = _batch(np.geomspace(19, 674, 31), 263, 300)
    db = api.Database.from_sequences(db_s)

    def least(**opts):
        x = []
        for _ in range(40):
            t = time.perf_counter()
            api.PreparedQueries(db, qs.residues, qs.offsets, BLOSUM62,
                                opts=api.options(band_stream="never", **opts)).close()
            x.append(time.perf_counter() - t)
        return min(x)

    try:
        assert least() < 5 * least(lanes_per_chain=16)
    finally:
        db.close()


@pytest.mark.parametrize("lens", [[31, 19, 674], [1, 2], [96, 97, 128, 129, 767, 768, 769], list(range(20, 660, 20)),
                                  list(range(3, 260))])
@pytest.mark.parametrize("mode", ["packed", "int32"])
@pytest.mark.parametrize("rows", [0, 4, 8, 12, 16, 24])
def test_scores_over_plans(api, lens, mode, rows):
    db_s, qs = _batch(lens, 37, 200)
    db = api.Database.from_sequences(db_s)
    try:
        batch = api.PreparedQueries(db, qs.residues, qs.offsets, BLOSUM62, mode=mode,
                                    opts=api.options(band_stream="never", rows_per_lane=rows))
        got = batch.search().cpu().numpy()
        batch.status()
        batch.close()
    finally:
        db.close()
    assert np.array_equal(got, oracle.scores(qs, db_s, BLOSUM62, 10, 2))
