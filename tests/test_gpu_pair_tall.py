"""The tallest bands that sw_align_pair picks by itself (28 rows per lane, two
warps per SM sub-partition, on 152 SMs) and those of long queries against short
targets, against 16- and 24-row bands of the same pair.  Scores are int32; the
bar is equality."""

import pytest

from workload import make_dna_pair
from workload.matrices import DNA_SUBMAT

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2412_08308_gb300 import api as _api
    from paper_2412_08308_gb300 import build

    build()
    return _api


@pytest.mark.parametrize("m,n,go,ge", [(1_000_000, 990_001, 5, 2), (1_000_001, 1_010_016, 4, 1), (2_000_001, 300, 5, 2),
                                       (400_000, 9_001, 4, 1), (1_000_000, 50_000, 5, 2)])
def test_tallest_bands(api, m, n, go, ge):
    query, target = make_dna_pair(m=m, n=n, seed=92)
    got = api.align_pair(query, target, DNA_SUBMAT, go, ge)
    assert got > 0
    for rows in (16, 24):
        assert got == api.align_pair(query, target, DNA_SUBMAT, go, ge, opts=api.pair_options(rows_per_lane=rows)), rows
