"""sw_search reads its results back in one copy up to 64 KB of scores and in
two above, and skips zeroing what a fresh upload has zeroed: same scores as a
prepared batch's at the sizes where the route changes, to host and device
memory, from several threads on their own streams at once (integers: equal)."""

import threading

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


def _case(rng, n_db, q_len):
    seqs = [rng.integers(0, 20, size=int(rng.integers(0, 70))).astype(np.uint8) for _ in range(n_db)]
    return from_list(seqs), from_list([rng.integers(0, 20, size=m).astype(np.uint8) for m in q_len])


def _expected(api, db, qs, mode):
    batch = api.PreparedQueries(db, qs.residues, qs.offsets, BLOSUM62, 10, 2, mode=mode)
    try:
        return batch.search().cpu().numpy()
    finally:
        batch.close()


@pytest.mark.parametrize("mode", ["packed", "int32"])
@pytest.mark.parametrize("n_db,q_len", [(1, [1]), (3, [60, 7, 1500]), (2048, [30] * 8), (2049, [30] * 8),
                                        (16383, [40]), (16384, [40]), (16385, [40])])
def test_host_and_device_results(api, n_db, q_len, mode):
    import torch

    s, qs = _case(np.random.Generator(np.random.PCG64(n_db)), n_db, q_len)
    db = api.Database(s.residues, s.offsets)
    try:
        exp = _expected(api, db, qs, mode)
        out = torch.empty((len(q_len), n_db), dtype=torch.int32, device="cuda")
        for _ in range(2):
            assert np.array_equal(api.search(db, qs.residues, qs.offsets, BLOSUM62, mode=mode), exp)
            api.search(db, qs.residues, qs.offsets, BLOSUM62, mode=mode, out=out.fill_(-1))
            assert np.array_equal(out.cpu().numpy(), exp)
    finally:
        db.close()


def test_threads_and_streams(api):
    import torch

    s, _ = _case(np.random.Generator(np.random.PCG64(5)), 900, [1])
    db = api.Database(s.residues, s.offsets)
    bad = []
    try:
        jobs = []
        for t in range(4):
            rng = np.random.Generator(np.random.PCG64(60 + t))
            for m in ([50], [300, 20], [1200]):
                qs = from_list([rng.integers(0, 20, size=k).astype(np.uint8) for k in m])
                jobs.append((t, qs, _expected(api, db, qs, "packed")))

        def work(t):
            stream = torch.cuda.Stream()
            for _ in range(20):
                for k, qs, exp in jobs:
                    if k == t and not np.array_equal(
                            api.search(db, qs.residues, qs.offsets, BLOSUM62, stream=stream), exp):
                        bad.append(t)

        threads = [threading.Thread(target=work, args=(t,)) for t in range(4)]
        for th in threads:
            th.start()
        for th in threads:
            th.join()
        assert not bad
    finally:
        db.close()
