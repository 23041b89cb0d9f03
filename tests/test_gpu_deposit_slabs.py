"""The tensor-core deposit at the edges of its slabs (16 particles), accumulation halves (96),
groups (192) and slab rotation (17 slabs), over one or many short work units, with particles
that carry no y between particles that do (the slab's y rows are zeroed once and kept)."""
import numpy as np
import pytest

from paper_2201_02632_gb300 import inputs as I
from tests.gpu_common import api, assigned_tensor, ctx, folded, orc_deposit_inputs  # noqa: F401
from tests.helpers import assert_map_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 15, 16, 17, 95, 96, 97, 191, 192, 193, 271, 272, 273, 289, 5000])
@pytest.mark.parametrize("unit", [256, 8192])
def test_slab_and_group_edges(orc, api, ctx, n, unit):
    nx, ny = 100, 70  # four tiles, ragged
    rng = np.random.default_rng(7000 + n)
    kind = np.where(np.arange(n) % 64 < 40, 1, 0)  # runs of field particles (no y)
    hp = rng.uniform(0.0, 60.0, n)
    hp[::11] = 0.0
    a = I.deposit_inputs(rng.uniform(-4, nx + 4, n), rng.uniform(-4, ny + 4, n), hp,
                         np.where(kind == 0, 10.0 ** rng.uniform(-9, -6, n), 0.0),
                         rng.normal(0, 1e-7, n), kind)
    ctx.set_tiling(pp_tile=64, pp_unit=unit)
    ctx.set_deposit_kernel("tensor")
    g = api.geom(nx, ny, 0.0, 0.0, 1.0)
    out = []
    for _ in range(2):
        maps = api.Maps.zeros(g)
        ctx.paste_particles(assigned_tensor(a), g, maps)
        out.append(folded(maps))
    yo, bo = orc.pp_deposit(orc_deposit_inputs(a), orc.geom(nx, ny, 0.0, 0.0, 1.0))
    if np.any(yo):
        assert_map_parity(out[0][0][0], yo, what="y")
    else:
        assert not np.any(out[0][0])
    # kSZ of both signs: relative to the map's norm
    b = out[0][1][0]
    assert np.linalg.norm(b - bo) <= 1e-5 * np.linalg.norm(bo)
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
