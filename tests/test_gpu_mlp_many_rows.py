"""The weight gradients of many rows in one call, against 64 bits.

Tolerance: a chain of L additions of terms of random sign in FP32 leaves about 2^-24 sqrt(L / 6)
of the sum (each addition rounds the partial sum, which grows as the root of its length).  512 rows
in a row: 5.5e-7, then 52 folds of a CTA and 152 CTAs: 6e-7 in all, the rest of a gradient 2e-7.
1.5e-6 allows twice that; one chain over all of a CTA's 26000 rows leaves up to 4e-6."""
import math

import pytest
import torch

from tests.gpu_common import api, ctx  # noqa: F401

pytestmark = pytest.mark.gpu
SIZES = ((6, 128), (128, 128), (128, 128), (128, 3))


def test_four_million_rows(api, ctx):
    n = 4_000_003
    g = torch.Generator(device="cuda")
    g.manual_seed(17)
    u = lambda *s: 2.0 * torch.rand(s, generator=g, device="cuda") - 1.0
    layers = [(math.sqrt(6.0 / (i + o)) * u(o, i), 0.1 * u(o)) for i, o in SIZES]
    P = torch.cat([t.reshape(-1) for l in layers for t in l])
    x = u(n, 6)
    dy = torch.randn((n, 3), generator=g, device="cuda")
    _, cache = ctx.mlp_forward(P, x)
    got = ctx.mlp_backward(P, x, cache, dy).double()
    del cache
    W = [(w.double(), b.double()) for w, b in layers]
    ref = torch.zeros_like(got)
    for xs, ds in zip(x.split(400_000), dy.split(400_000)):
        A, Z, d, out = [xs.double()], [], ds.double(), []
        for w, b in W[:3]:
            Z.append(A[-1] @ w.T + b)
            A.append(0.5 * Z[-1] * (1.0 + torch.erf(Z[-1] / math.sqrt(2.0))))
        for k in (3, 2, 1, 0):
            out = [(d.T @ A[k]).reshape(-1), d.sum(0)] + out
            if k:
                z = Z[k - 1]
                d = (d @ W[k][0]) * (0.5 * (1.0 + torch.erf(z / math.sqrt(2.0))) +
                                     z * torch.exp(-0.5 * z * z) / math.sqrt(2.0 * math.pi))
        ref += torch.cat(out)
    err = float((got - ref).norm() / ref.norm())
    print(f"relative error {err:.2e}")
    assert err <= 1.5e-6
