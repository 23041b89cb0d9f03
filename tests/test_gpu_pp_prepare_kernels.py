"""A pair list prepared for one deposit kernel, deposited by another: bp_pp_deposit asks for the
same records, geometry and selection, not for the kernel that bp_set_deposit_kernel named before.

Tolerance: that of every map comparison with the oracle (assert_map_parity)."""
import numpy as np
import pytest

from paper_2201_02632_gb300 import inputs as I
from tests.gpu_common import api, assigned_tensor, ctx, folded, orc_deposit_inputs  # noqa: F401
from tests.helpers import assert_map_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("first,then", [("tensor", "simt"), ("simt", "tensor"), ("auto", "simt"),
                                        ("simt", "simt"), ("tensor", "tensor")])
@pytest.mark.parametrize("unit", [0, 256])
def test_prepared_by_one_kernel_deposited_by_another(orc, api, ctx, first, then, unit):
    nx, ny, n = 150, 97, 3000
    rng = np.random.default_rng(77)
    a = I.deposit_inputs(rng.uniform(0, nx, n), rng.uniform(0, ny, n), rng.uniform(0.0, 12.0, n),
                         10.0 ** rng.uniform(-9, -6, n), rng.normal(0, 1e-7, n),
                         rng.integers(0, 2, n))
    a["Y"] = np.where(a["kind"] == api.KIND_FIELD, 0.0, a["Y"])
    g = api.geom(nx, ny, 0.0, 0.0, 1.0)
    rec, maps = assigned_tensor(a), api.Maps.zeros(g)
    if unit:
        ctx.set_tiling(pp_unit=unit)  # tiles split into several units
    ctx.set_deposit_kernel(first)
    ctx.pp_prepare(rec, g)
    ctx.set_deposit_kernel(then)
    ctx.pp_deposit(rec, g, maps)
    y, b = folded(maps)
    yo, bo = orc.pp_deposit(orc_deposit_inputs(a), orc.geom(nx, ny, 0.0, 0.0, 1.0))
    assert_map_parity(y[0], yo, what="y")
    assert np.linalg.norm(b[0] - bo) <= 1e-5 * np.linalg.norm(bo)
