"""All-sky HP maps at the edges of the ring segments (256 pixels): nside around the multiples of
64 where a cap ring gains a segment, and odd ones; apertures from a pixel (values stored per
pixel) to hundreds (tables), on the poles and across phi = 0.

Tolerance: the map's relative L2 bound.  Single pixels are not compared: among the 1e4 pixels of
a near halo's aperture the outermost has 1 - u of about 1e-4, where the chord sqrt(1 - u^2)
turns the FP32 rounding of u into 1e-7 / (2e-4) = 5e-4 of the pixel."""
import numpy as np
import pytest

from paper_2201_02632_gb300 import inputs as I
from tests.gpu_common import api, ctx, cuda  # noqa: F401
from tests.helpers import MAP_REL_L2, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside", [1, 3, 63, 64, 65, 129])
def test_segments_around_cap_rings(orc, api, ctx, nside):
    far = I.allsky_catalog(60, seed=I.SEED_BASE + nside, logm=(13.5, 14.5), zr=(0.3, 1.0),
                           volume=False, n_polar=4)
    near = I.allsky_catalog(40, seed=I.SEED_BASE + 500 + nside, logm=(14.0, 15.3),
                            zr=(0.005, 0.05), volume=False, n_polar=4)
    cat = {k: np.concatenate([far[k], near[k]]) for k in ("M", "c", "z", "theta", "phi", "vlos")}
    cat["phi"][:4] = np.array([0.0, 1e-4, 2 * np.pi - 1e-4, 2 * np.pi])
    model, status = ctx.solve_halos(cuda(cat["M"]), cuda(cat["c"]), cuda(cat["z"]))
    maps = api.healpix_maps(nside)
    ctx.paste_halos_healpix(cuda(cat["theta"]), cuda(cat["phi"]), cuda(cat["vlos"]), model, status,
                            nside, maps)
    mo = orc.solve_halos(cat["M"], cat["c"], cat["z"])
    pt, pp = orc.hpx_centres(nside, None)
    yo, bo = orc.hp_sky(cat["theta"], cat["phi"], cat["vlos"], mo, pt, pp, ap_r500=0.0, rtol=1e-9)
    for a, lo, o, what in ((maps.y, maps.ylo, yo, "y"), (maps.b, maps.blo, bo, "b")):
        got = a.double().cpu().numpy().ravel() + lo.double().cpu().numpy().ravel()
        assert rel_l2(got, o) <= MAP_REL_L2, what
