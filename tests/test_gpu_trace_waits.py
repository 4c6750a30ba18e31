"""A traceback whose wait between two bands expires: the fill stops, bands that
were not taken leave no best cell, and the walk must not follow what their
memory held before.  The call reports SW_ETIMEOUT and the context stays usable."""

import ctypes

import numpy as np
import pytest

import oracle
from workload import random_sequences
from workload.matrices import BLOSUM62

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2412_08308_gb300 import api as _api
    from paper_2412_08308_gb300 import build

    build()
    oracle.build()
    return _api


def test_expired_wait_ends_the_traceback(api):
    import torch

    from paper_2412_08308_gb300 import _native as N

    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    for budget in (1, 1000, 5000):
        assert N.sw_selftest_trace(budget, s) == (N.SW_ETIMEOUT, -1)
    # the same hit with time to finish
    assert N.sw_selftest_trace(1 << 33, s) == (N.SW_OK, 16)
    # the same process aligns on
    seqs, qs = random_sequences(83, 6, 300, 0.5, 40, 700), random_sequences(84, 2, 600, 0.2, 400, 800)
    hits = [(i, j) for i in range(2) for j in range(6)]
    db = api.Database.from_sequences(seqs)
    got = api.traceback(db, qs.residues, qs.offsets, hits, BLOSUM62)
    db.close()
    for (i, j), g in zip(hits, got):
        assert g == oracle.align(qs[i], seqs[j], BLOSUM62, 10, 2)
    assert np.all([g[0] > 0 for g in got])


@pytest.mark.parametrize("budget", [0, -1, (1 << 36) + 1])
def test_invalid_budget(api, budget):
    from paper_2412_08308_gb300 import _native as N

    with pytest.raises(N.SwError) as e:
        N.sw_selftest_trace(budget, ctypes.c_void_p(0))
    assert e.value.code == N.SW_EINVAL
