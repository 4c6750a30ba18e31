"""Single-call searches from several threads on streams of their own: every
round of every thread must end, with the oracle's scores (an exception in a
thread fails the test)."""

from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

import oracle
from workload import from_list
from workload.matrices import BLOSUM62

pytestmark = pytest.mark.gpu

ROUNDS = 20


@pytest.fixture(scope="module")
def api():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2412_08308_gb300 import api as _api
    from paper_2412_08308_gb300 import build

    build()
    oracle.build()
    return _api


@pytest.mark.parametrize("mode", ["packed", "int32"])
def test_every_round_of_every_thread(api, mode):
    import torch

    rng = np.random.Generator(np.random.PCG64(6))
    # (4 queries x 5,000 sequences: scores past the 64 KB that come back with the status words)
    dbs = [from_list([rng.integers(0, 20, size=int(k)).astype(np.uint8) for k in rng.integers(0, hi, size=n)])
           for n, hi in ((900, 70), (5000, 25))]
    handles = [api.Database.from_sequences(d) for d in dbs]
    jobs = [[] for _ in range(4)]
    for t in range(4):
        for lens in ([50], [300, 20], [1200], [9, 30, 30, 61]):
            qs = from_list([rng.integers(0, 20, size=k).astype(np.uint8) for k in lens])
            for d, h in zip(dbs, handles):
                jobs[t].append((h, qs, oracle.scores(qs, d, BLOSUM62, 10, 2)))

    def work(t):
        stream, done = torch.cuda.Stream(), 0
        for _ in range(ROUNDS):
            for h, qs, exp in jobs[t]:
                got = api.search(h, qs.residues, qs.offsets, BLOSUM62, mode=mode, stream=stream)
                assert np.array_equal(got, exp), (t, done)
                done += 1
        return done

    try:
        with ThreadPoolExecutor(4) as ex:
            done = [f.result() for f in [ex.submit(work, t) for t in range(4)]]
    finally:
        for h in handles:
            h.close()
    assert done == [ROUNDS * len(j) for j in jobs]
