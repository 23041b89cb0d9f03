"""Smoothing lengths at the edges of the search tree and of its groups: particle counts around
whole leaves (32) and nodes (1024), the largest N_ngb of the group kernel and the next one, and
kernels with a dense clump at their edge, whose candidates overflow a list.

Tolerance: N_eff sums at most 128 weights one after the other per lane, then a tree of 5 adds
(relative error below 4e-6, all weights positive), Newton leaves 2e-7, and N_eff grows like h^3:
1e-5 relative in h holds with a margin."""
import numpy as np
import pytest

from paper_2201_02632_gb300 import inputs as I
from tests.gpu_common import api, ctx, cuda  # noqa: F401

pytestmark = pytest.mark.gpu
RTOL = 1e-5


def _gpu(ctx, p, n_ngb):
    return ctx.smoothing_lengths(cuda(p[0]), cuda(p[1]), cuda(p[2]), n_ngb).double().cpu().numpy()


@pytest.mark.parametrize("n", [7, 31, 32, 33, 63, 65, 1023, 1024, 1025, 2049])
def test_counts_around_leaves_and_nodes(orc, api, ctx, n):
    p = np.random.default_rng(n).normal(0.0, 2.0, (3, n)).astype(np.float32)
    k = min(32.0, 5.0 * n)
    np.testing.assert_allclose(_gpu(ctx, p, k), orc.smoothing_lengths(*p, k), rtol=RTOL)


@pytest.mark.parametrize("n_ngb", [11.0, 127.5, 128.0, 129.0])
def test_neighbour_numbers_around_the_groups(orc, api, ctx, n_ngb):
    p = np.random.default_rng(5).uniform(0.0, 9.0, (3, 3001)).astype(np.float32)
    np.testing.assert_allclose(_gpu(ctx, p, n_ngb), orc.smoothing_lengths(*p, n_ngb), rtol=RTOL)


@pytest.mark.parametrize("clump", [150, 1500, 9000])
def test_clumps_at_the_edge_of_kernels(orc, api, ctx, clump):
    rng = np.random.default_rng(I.SEED_BASE + clump)
    field = rng.uniform(-10.0, 10.0, (3, 1500))
    dense = rng.normal(0.0, 0.02, (3, clump)) + rng.uniform(-6.0, 6.0, (3, 1))
    p = np.concatenate([field, dense], axis=1).astype(np.float32)
    idx = np.concatenate([np.arange(1500), 1500 + rng.choice(clump, 40, replace=False)])
    np.testing.assert_allclose(_gpu(ctx, p, 64.0)[idx], orc.smoothing_lengths_at(*p, idx, 64.0),
                               rtol=RTOL)
