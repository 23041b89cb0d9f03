"""Maps of few rows (several columns per CTA in the second transform) with few and many bins,
against the oracle with the tolerance of test_gpu_spectrum, and their time."""
import math

import numpy as np
import pytest
import torch

from tests.gpu_common import api, ctx  # noqa: F401
from tests.test_gpu_spectrum import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny", [2, 4, 16, 64, 256, 512])
@pytest.mark.parametrize("nb", [1, 30, 200, 256])
def test_short_columns(orc, api, ctx, ny, nb):
    nx, d = 64, 1e-4
    m = np.random.default_rng(ny + nb).normal(size=(ny, nx)) + 1.0
    edges = np.concatenate([[0.0], np.geomspace(math.pi / (max(nx, ny) * d), 2 * math.pi / d, nb)])
    _, cnt = _check(orc, api, ctx, m, d, edges)
    if nb > 1:  # (one bin ends at the first edge)
        assert cnt.sum() == nx * ny


def test_few_rows_cost_little(api, ctx):
    """A 512 x 2 map takes less than 3 times a 512 x 512 one (11 times with a warp per column and
    bin, 1.2 times with a thread)."""
    def us(ny):
        m = torch.randn((ny, 512), device="cuda")
        best = float("inf")
        for _ in range(10):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            for _ in range(10):
                ctx.power_spectrum(m, 1e-4)
            b.record()
            torch.cuda.synchronize()
            best = min(best, 100.0 * a.elapsed_time(b))
        return best

    few, many = us(2), us(512)
    print(f"512 x 2 {few:.0f} us, 512 x 512 {many:.0f} us")
    assert few <= 3.0 * many
