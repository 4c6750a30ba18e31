"""Long queries against many peptides: a band's last lane ends every unit 31
columns after its first, so band-stream jobs cost a peptide twice its cells and
more.  The default plan is near the faster side; scores stay the same."""

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


def _compare(api, n, lo, hi, q_len, mode, long=()):
    """Least device time (ms) of the default plan and of the other two; equal scores."""
    import torch

    rng = np.random.Generator(np.random.PCG64(n + hi))
    lens = np.concatenate([rng.integers(lo, hi + 1, size=n), np.array(long, dtype=np.int64)])
    res = rng.integers(0, 20, size=int(lens.sum())).astype(np.uint8)
    qs = from_list([rng.integers(0, 20, size=k).astype(np.uint8) for k in q_len])
    db = api.Database(res, np.concatenate([[0], np.cumsum(lens)]))
    got, ms = [], []
    try:
        for band in ("auto", "never", "always"):
            batch = api.PreparedQueries(db, qs.residues, qs.offsets, BLOSUM62, mode=mode,
                                        opts=api.options(band_stream=band))
            out = batch.search()
            times = []
            for _ in range(12):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                batch.search(out)
                b.record()
                b.synchronize()
                times.append(a.elapsed_time(b))
            ms.append(min(times))
            got.append(out.cpu().numpy())
            batch.status()
            batch.close()
    finally:
        db.close()
    assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2])
    return ms


# (the slower side took 2.1 times the other's)
@pytest.mark.parametrize("n,q_len,mode,long", [(16000, [3783, 4557], "int32", []), (57000, [4852], "int32", [4852] * 3),
                                               (16000, [4557], "packed", [])])
def test_long_queries_against_peptides(api, n, q_len, mode, long):
    auto, never, always = _compare(api, n, 10, 40, q_len, mode, long)
    assert auto < 1.5 * min(never, always), (auto, never, always)


# more than 16,384 short sequences (inter-task alone: 1.7 to 2.1 times the transposed jobs' time)
@pytest.mark.parametrize("n,lo,hi,q_len", [(17000, 1, 200, [300]), (60000, 1, 60, [800]), (60000, 1, 60, [1000])])
@pytest.mark.parametrize("mode", ["packed", "int32"])
def test_many_short_sequences(api, n, lo, hi, q_len, mode):
    auto, never, always = _compare(api, n, lo, hi, q_len, mode, [1000])
    assert auto < 1.4 * min(never, always), (auto, never, always)


# the edges of the rule: 16,384 sequences, 200 residues on average, 10 million together
@pytest.mark.parametrize("n,length", [(16384, 200), (16385, 200), (16385, 201), (50000, 200), (50001, 200)])
@pytest.mark.parametrize("q_len", [[1], [59, 61], [300], [1024]])
@pytest.mark.parametrize("mode", ["packed", "int32"])
def test_edges_of_the_rule(api, n, length, q_len, mode):
    _compare(api, n, length, length, q_len, mode)
