"""The order in which the bands of transposed jobs are handed out: job by job or
by level, with up to more levels than a warp has lanes, sequences of very
different lengths, one query and many.  Scores against the inter- and
intra-task kernels' (integers: equal)."""

import numpy as np
import pytest

from workload import from_list
from workload.matrices import BLOSUM62

pytestmark = pytest.mark.gpu

# database lengths (count, length), query lengths: levels and order of the 16-row lanes' bands
CASES = {
    "one_level": ([(200, 300)], [50]),
    "two_levels": ([(200, 300), (50, 700)], [50, 144]),
    "three_levels_job_by_job": ([(100, 300), (60, 1100), (20, 900)], [1000]),
    "three_levels_by_level": ([(100, 300), (60, 1100), (20, 900)], [60]),
    "many_jobs": ([(300, 300), (300, 1500), (100, 2500)], [100, 200, 300, 400, 500, 600]),
    "deep": ([(7, 20000), (2, 9000), (30, 40), (1, 2049)], [144]),
    "deep_many_queries": ([(5, 20000), (3, 1025), (40, 200)], [90 + 3 * k for k in range(40)]),
    "equal_depths": ([(64, 1500)], [17] * 33),
    "one_sequence": ([(1, 17500)], [1]),
}


@pytest.fixture(scope="module")
def api():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2412_08308_gb300 import api as _api
    from paper_2412_08308_gb300 import build

    build()
    return _api


@pytest.mark.parametrize("case", list(CASES))
@pytest.mark.parametrize("mode", ["packed", "int32"])
def test_orders_agree(api, case, mode):
    lens, q_len = CASES[case]
    rng = np.random.Generator(np.random.PCG64(sum(q_len)))
    seqs = [rng.integers(0, 20, size=L).astype(np.uint8) for n, L in lens for _ in range(n)]
    qs = [rng.integers(0, 20, size=m).astype(np.uint8) for m in q_len]
    for k, q in enumerate(qs[:3]):  # (some alignments longer than chance gives, across bands)
        s = seqs[(5 * k) % len(seqs)]
        at = max(0, min(len(s) - len(q), 500 + 7 * k))
        s[at:at + len(q)] = q[:len(s) - at]
    db, qs = api.Database.from_sequences(from_list(seqs)), from_list(qs)
    try:
        got = []
        for band in ("always", "never"):
            # (band_rows 16: a query below 1,024 residues runs transposed)
            batch = api.PreparedQueries(db, qs.residues, qs.offsets, BLOSUM62, mode=mode,
                                        opts=api.options(band_stream=band))
            got.append(batch.search().cpu().numpy())
            batch.status()
            batch.close()
    finally:
        db.close()
    assert np.array_equal(got[0], got[1])


# one or a few sequences past the length from which packed mode may take int32 tracks
@pytest.mark.parametrize("lens", [[(1, 20000)], [(300, 300), (1, 2048), (1, 2049), (2, 9000)], [(300, 300), (1, 35000)],
                                  [(40, 4000)], [(400, 2500)]])
@pytest.mark.parametrize("q_len", [[60], [400], [144, 700], [1500]])
def test_deep_sequences_in_either_width(api, lens, q_len):
    rng = np.random.Generator(np.random.PCG64(len(lens) + len(q_len)))
    seqs = [rng.integers(0, 20, size=L).astype(np.uint8) for n, L in lens for _ in range(n)]
    qs = [rng.integers(0, 20, size=m).astype(np.uint8) for m in q_len]
    seqs[-1][1000:1000 + len(qs[0])] = qs[0][:len(seqs[-1]) - 1000]
    db, qs = api.Database.from_sequences(from_list(seqs)), from_list(qs)
    try:
        got = []
        for opts in (None, api.options(band_stream="always"), api.options(band_stream="never")):
            batch = api.PreparedQueries(db, qs.residues, qs.offsets, BLOSUM62, mode="packed", opts=opts)
            got.append(batch.search().cpu().numpy())
            batch.status()
            batch.close()
    finally:
        db.close()
    assert np.array_equal(got[0], got[2]) and np.array_equal(got[1], got[2])
