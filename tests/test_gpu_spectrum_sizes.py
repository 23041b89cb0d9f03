"""The power spectrum at every transform length (2 .. 8192 points along each axis: all first
radices and pass counts), against the oracle with the tolerance of test_gpu_spectrum."""
import math

import numpy as np
import pytest

from paper_2201_02632_gb300 import inputs as I
from tests.gpu_common import api, ctx  # noqa: F401
from tests.test_gpu_spectrum import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lgx,lgy", [(k, 14 - k) for k in range(1, 14)] + [(1, 1), (13, 3), (2, 13)])
def test_every_length(orc, api, ctx, lgx, lgy):
    nx, ny = 1 << lgx, 1 << lgy
    rng = np.random.default_rng(I.SEED_BASE + 100 * lgx + lgy)
    d = 3e-5
    m = rng.normal(size=(ny, nx)) + 3.0
    lo = 1e-8 * rng.normal(size=(ny, nx))
    # narrow bins from zero up: bins that hold one mode, none, and the axes' own modes
    edges = np.concatenate([[0.0], np.geomspace(2 * math.pi / (max(nx, ny) * d) * 0.5,
                                                2 * math.pi / d, 64)])
    _, cnt = _check(orc, api, ctx, m, d, edges, lo=lo if lgx % 2 else None)
    assert cnt.sum() == nx * ny  # no |l| beyond the last edge
