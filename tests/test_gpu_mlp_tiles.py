"""The FP32 training kernels at the edges of their 32-row tiles and of one tile per SM, and with
parameters that are not 16-byte aligned, against the FP64 CPU MLP (same tolerances as the
whole-network test)."""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp
from tests.gpu_common import api, ctx, cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 32, 33, 4863, 4865, 20001])
@pytest.mark.parametrize("shift", [0, 1])
def test_forward_backward_tiles(api, ctx, n, shift):
    rng = np.random.default_rng(100 + n)
    n_par = sum(a * b + b for a, b in omlp.SIZES)
    p = rng.normal(0, 0.15, n_par).astype(np.float32)
    x = rng.uniform(-1, 1, (n, 6)).astype(np.float32)
    dy = rng.normal(0, 1, (n, 3)).astype(np.float32)
    P = torch.empty(n_par + shift, device="cuda")[shift:]
    P.copy_(cuda(p))
    y, cache = ctx.mlp_forward(P, cuda(x))
    g = ctx.mlp_backward(P, cuda(x), cache, cuda(dy))
    yo, co = omlp.forward(p.astype(np.float64), x.astype(np.float64))
    go = omlp.backward(p.astype(np.float64), co, dy.astype(np.float64))
    np.testing.assert_allclose(y.cpu().numpy(), yo, rtol=1e-4, atol=1e-5)
    gg = g.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(gg - go) <= 2e-4 * np.linalg.norm(go)
    # every layer's block of the gradient by itself
    off = 0
    for a, b in omlp.SIZES:
        for k in (a * b, b):
            s = slice(off, off + k)
            assert np.linalg.norm(gg[s] - go[s]) <= 2e-4 * np.linalg.norm(go[s])
            off += k
