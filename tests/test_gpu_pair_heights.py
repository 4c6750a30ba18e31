"""Band heights that sw_align_pair picks by itself (4 to 28 rows per lane, one
or two warps per SM sub-partition, several rounds of bands): each against the
16-row bands of the same pair, and against the pair with its roles exchanged
(another height, other rings; the DNA matrix is symmetric).  Scores are int32;
the bar is equality.
"""

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


# (on 152 SMs: 4, 6, 8, 10, 12, 14, 16, 20, 24, 28 rows per lane; 512 and 513
# columns end on and just past a staged chunk of residues)
@pytest.mark.parametrize("m,n", [(20_001, 25_003), (100_000, 60_000), (125_000, 120_000), (162_000, 172_000),
                                 (230_000, 200_000), (270_000, 250_000), (300_000, 310_000), (380_000, 380_000),
                                 (460_000, 400_000), (100_000, 2_000), (70_000, 512), (70_000, 513)])
@pytest.mark.parametrize("go,ge", [(5, 2), (4, 1)])
def test_picked_height(api, m, n, go, ge):
    query, target = make_dna_pair(m=m, n=n, seed=91)
    got = api.align_pair(query, target, DNA_SUBMAT, go, ge)
    assert got > 0
    assert got == api.align_pair(query, target, DNA_SUBMAT, go, ge, opts=api.pair_options(rows_per_lane=16))
    assert got == api.align_pair(target, query, DNA_SUBMAT, go, ge)
