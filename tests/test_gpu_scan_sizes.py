"""Work lists of particle counts around the scans' limits (one block up to 16384 counts, chunks of
8192 after that, 16-byte accesses where a thread's eight counts are whole): every particle has to
arrive in the maps, exactly as often as the oracle's.

Tolerance: that of every map comparison with the oracle (assert_map_parity)."""
import numpy as np
import pytest

from paper_2201_02632_gb300 import inputs as I
from tests.gpu_common import api, assigned_tensor, ctx, folded, orc_deposit_inputs  # noqa: F401
from tests.helpers import assert_map_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8191, 8193, 16383, 16384, 16385, 24575, 24577, 32769])
def test_counts_around_scan_chunks(orc, api, ctx, n):
    nx, ny = 130, 65
    rng = np.random.default_rng(9000 + n)
    a = I.deposit_inputs(rng.uniform(0, nx, n), rng.uniform(0, ny, n), rng.uniform(0.0, 3.0, n),
                         10.0 ** rng.uniform(-9, -6, n), rng.normal(0, 1e-7, n),
                         np.ones(n, np.int64))
    g = api.geom(nx, ny, 0.0, 0.0, 1.0)
    maps = api.Maps.zeros(g)
    ctx.paste_particles(assigned_tensor(a), g, maps)
    y, b = folded(maps)
    yo, bo = orc.pp_deposit(orc_deposit_inputs(a), orc.geom(nx, ny, 0.0, 0.0, 1.0))
    assert_map_parity(y[0], yo, what="y")
    assert np.linalg.norm(b[0] - bo) <= 1e-5 * np.linalg.norm(bo)
