"""The power spectrum's rounding, against an extended-precision transform.

Tolerance: a correctly rounded mean leaves 6.4e-17 rms (uniform within half a unit in the last
place, over all mantissas); the bins' sums and the transforms' errors, averaged over the hundreds
of modes of a bin, about as much again: 8e-17 to 9e-17.  1.05e-16 rms allows a fifth more.  A
modulus of the twiddles 7e-17 above 1 in each direction, or a second rounding of the mean, is
beyond it."""
import numpy as np
import pytest
import scipy.fft
import torch

from tests.gpu_common import api, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


def test_bins_of_a_white_map(api, ctx):
    nx, ny, nb, d = 4096, 512, 200, 2e-5
    if np.finfo(np.longdouble).eps > 2e-19:
        pytest.skip("no extended precision here")
    edges = np.linspace(1.0, np.pi / d, nb + 1)
    l2 = ((2 * np.pi * np.fft.rfftfreq(nx, d))[None] ** 2 +
          (2 * np.pi * np.fft.fftfreq(ny, d))[:, None] ** 2).ravel()
    b = np.searchsorted(edges ** 2, l2, side="right") - 1
    use = (b >= 0) & (b < nb)
    weight = np.full(nx // 2 + 1, 2)
    weight[[0, -1]] = 1
    weight = np.broadcast_to(weight, (ny, weight.size)).ravel()
    count = np.bincount(b[use], weights=weight[use], minlength=nb)
    err = []
    for seed in range(2):
        m = np.random.default_rng(seed).standard_normal((ny, nx)).astype(np.float32)
        _, cl, modes = ctx.power_spectrum(torch.from_numpy(m).cuda(), d, edges=edges)
        f = scipy.fft.rfft2(m.astype(np.longdouble), workers=8)
        p = (f.real ** 2 + f.imag ** 2).ravel() * (np.longdouble(d) ** 2 / (nx * ny)) * weight
        ref = np.zeros(nb, np.longdouble)
        np.add.at(ref, b[use], p[use])
        same = modes.cpu().numpy() == count  # (a mode on an edge may be taken either way)
        assert same.sum() > 0.9 * nb
        err.append((cl.cpu().numpy()[same] / (ref[same] / count[same]) - 1).astype(float))
    err = np.concatenate(err)
    print(f"rms {np.sqrt((err ** 2).mean()):.3e}, mean {err.mean():.2e}")
    assert np.sqrt((err ** 2).mean()) <= 1.05e-16
