"""The one-thread-per-halo pre-solve and Newton: concentrations on and beside the edges of their
tabulated quadrature panels (0.5 x 2.5^k) against the oracle, and the independence of a halo's
solution from its place in the launch."""
import numpy as np
import pytest
import torch

from tests.gpu_common import api, ctx, cuda  # noqa: F401
from tests.test_gpu_solve import _compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("icm", [dict(), dict(energy_sign=1), dict(Gamma=1.15)])
def test_panel_edges(orc, api, icm):
    edges = 0.5 * 2.5 ** np.arange(1, 5)  # 1.25 .. 19.5
    cc = np.concatenate([edges * f for f in (1 - 1e-9, 1.0, 1 + 1e-9, 1.3)])
    M = np.concatenate([np.full(cc.size, 1e13), np.full(cc.size, 8e14)])
    c = np.concatenate([cc, cc])
    z = np.linspace(0.02, 2.9, c.size)
    ctx = api.Context(icm=icm)
    mo = orc.solve_halos(M, c, z, ip=orc.icm_default(**icm))
    model, status = ctx.solve_halos(cuda(M), cuda(c), cuda(z), raise_on_noconv=False)
    ok = mo[:, orc.F["status"]] == 0
    assert ok.sum() > 0.8 * ok.size
    assert np.array_equal(status.cpu().numpy() == 0, ok)
    _compare(orc, api, mo[ok], model.cpu().numpy()[:, ok])
    torch.cuda.synchronize()
    ctx.close()


@pytest.mark.parametrize("k", [1, 31, 33, 129, 5000])
def test_independent_of_the_launch(api, ctx, k):
    rng = np.random.default_rng(91)
    n = 25000  # blocks of 128; the short launches use one warp per block
    M, c, z = 10 ** rng.uniform(12, 15.3, n), rng.uniform(1.5, 20, n), rng.uniform(0.01, 3, n)
    full, st = ctx.solve_halos(cuda(M), cuda(c), cuda(z), raise_on_noconv=False)
    part, sp = ctx.solve_halos(cuda(M[:k]), cuda(c[:k]), cuda(z[:k]), raise_on_noconv=False)
    assert torch.equal(part, full[:, :k].contiguous()) and torch.equal(sp, st[:k])
