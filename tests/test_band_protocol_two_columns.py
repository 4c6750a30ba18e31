"""The pair kernel's boundary protocol as its two-column steps run it (no GPU):
the model of test_band_protocol.py with rows stored 64 columns behind the first
lane, two at a time, and consumed columns handed back every up to 128 blocks.
Rings past 2,048 columns make the larger interval matter."""

import os
import re

import pytest

from . import test_band_protocol as model
from .test_band_protocol import COL, Band, Sim

LAG = 64  # 32 lanes x 2 columns (the store is one step behind the last lane's)
CAP = 128  # blocks between hand-backs, at most


class TwoColumnSim(Sim):
    def __init__(self, npad, nbands, gw, ring_columns, seed):
        super().__init__(npad, nbands, gw, LAG, ring_columns, seed)
        self.cons_every = max(1, min(CAP, self.window // COL // 8))


class PairedBand(Band):
    def write(self, t0, t1):
        assert (t1 - t0) % 2 == 0 and (t0 - self.sim.lag) % 2 == 0  # whole pairs of columns
        super().write(t0, t1)


@pytest.mark.parametrize("npad,nbands,gw,ring", [
    (16, 3, 1, 0), (256, 7, 3, 0), (1008, 13, 4, 256), (2000, 9, 2, 256), (4096, 24, 5, 0), (1600, 30, 3, 512),
    (9600, 7, 2, 2064), (12288, 9, 3, 4096), (20000, 5, 2, 8192), (40000, 4, 1, 16384)])
def test_two_column_protocol(monkeypatch, npad, nbands, gw, ring):
    monkeypatch.setattr(model, "Band", PairedBand)
    for seed in range(2):
        TwoColumnSim(npad, nbands, gw, ring, seed=1000 * seed + npad + nbands).run()


def test_model_follows_the_host():
    # the hand-back cap and the store's lag as the sources have them
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    csrc = os.path.join(root, "paper_2412_08308_gb300", "csrc")
    pair = open(os.path.join(csrc, "pair.cu")).read()
    assert int(re.search(r"cons_every = .*std::min<int64_t>\((\d+), window / kColBlock / 8\)", pair).group(1)) == CAP
    cols = int(re.search(r"constexpr int kPairCols = (\d+);", open(os.path.join(csrc, "k_pair.cu")).read()).group(1))
    assert re.search(r"constexpr int kStoreLagBlocks = 32 \* COLS / kColBlock;",
                     open(os.path.join(csrc, "band_core.cuh")).read())
    assert 32 * cols == LAG
