"""Bright pixels behind large read noise, and the smallest expected images.

With 4e5..4e6 photons a pixel and a read noise of as many photons^2 the photon
posterior spreads over 4.5e2..1.4e3 counts, so a sum to 2^-56 of its mode runs over
up to 12 000 counts on either side.  The log posterior is compared with the
oracle's Eq. 9 (whose sums have no such bound), likelihood changes with a sum in
double over 14 standard deviations whose terms are ratios to the mode's."""
import math

import numpy as np
import pytest

from oracle import oracle as O
from paper_2411_00991_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2411_00991_gb300 import bdecon  # noqa: E402


def _problem(level, n=10):
    rng = np.random.default_rng(int(level))
    mu = level * np.exp(0.05 * rng.standard_normal((n, n)))
    img = (rng.poisson(mu) + rng.normal(size=(n, n)) * math.sqrt(level)).astype(np.float32)
    return mu, synth.Problem(image=img, psf=np.ones((1, 1)), gain=1.0, offset=0.0, var=float(level), stride=1, seed=1,
                             refresh_every=0)


def _change(c, is2, m, x):
    """l(m + x) - l(m): ratios to the term of the count nearest m (to 14 deviations past either sum's mode)."""
    f0, w = int(round(m)), int(14 * math.sqrt(m) + abs(x))
    up = np.arange(f0, f0 + w)
    dn = np.arange(f0, max(0, f0 - w), -1)
    lu = np.cumsum(is2 * (c - up - 0.5) + np.log(m / (up + 1.0)))
    ld = np.cumsum(-is2 * (c - dn + 0.5) + np.log(dn / m))
    k = np.concatenate([[0], up + 1 - f0, dn - 1 - f0]).astype(float)
    t = np.concatenate([[0.0], lu, ld])
    r = math.log1p(x / m)
    v = t + k * r
    return (math.log(np.exp(v - v.max()).sum()) + v.max() - math.log(np.exp(t - t.max()).sum()) - t.max()) + (f0 * r - x)


@pytest.mark.parametrize("precision", [bdecon.BDECON_FP64, bdecon.BDECON_FP32])
@pytest.mark.parametrize("level", [4e5, 4e6])
def test_log_posterior_of_bright_noisy_frames(level, precision):
    mu, p = _problem(level)
    s = bdecon.Sampler(p, precision=precision, max_sweeps=4)
    s.set_state(mu.astype(np.float32).astype(np.float64), 0)
    ref = O.Oracle(p).log_posterior(s.get_state()[0])
    # a term of the sums rounds at 1e-16 of the counts times their logarithms
    assert abs(s.log_posterior() - ref) <= 1e-15 * level * 16 * mu.size
    s.close()


@pytest.mark.parametrize("level", [4e5, 4e6])
def test_likelihood_changes_of_bright_noisy_pixels(level):
    mu, p = _problem(level)
    s = bdecon.Sampler(p, precision=bdecon.BDECON_FP64, max_sweeps=4)
    s.set_state(mu, 0)
    for i in (0, 17, 99):
        for d in (-0.02, -1e-3, 1e-4, 1e-3, 5e-3, 0.02):
            m = float(mu.flat[i])
            new = m * (1 + d)
            ok, dl, _ = s.delta(i, new)
            ref = _change(float(p.image.flat[i]), 1.0 / level, m, new - m)
            # 28 sqrt(level) terms' logarithms, and the difference of terms of the size of |new - m|
            assert ok and abs(dl - ref) <= 1e-12 * abs(new - m) + 1e-16 * 28 * math.sqrt(level) * level ** 0.5, (i, d, dl, ref)
    s.close()


def test_log_posterior_at_the_smallest_expected_image():
    rng = np.random.default_rng(3)
    # an offset of a photon too much, 0.03 photons of read noise: the first ratio of
    # the terms below the mode, which is 0 and has none, overflows
    img = (0.01 * rng.normal(size=(6, 7)) - 1.0).astype(np.float32)
    p = synth.Problem(image=img, psf=np.ones((1, 1)), gain=1.0, offset=0.0, var=1e-3, stride=1, seed=1, refresh_every=0)
    s = bdecon.Sampler(p, precision=bdecon.BDECON_FP64, max_sweeps=4)
    for v in (1e-10, 1e-120, 1e-140):
        rho = np.full((6, 7), v) * (1 + 0.01 * rng.random((6, 7)))
        s.set_state(rho, 0)
        ref = O.Oracle(p).log_posterior(rho)
        assert abs(s.log_posterior() - ref) <= 1e-12 * abs(ref)
        new = 1.1 * rho.flat[5]
        ok, dl, _ = s.delta(5, new)
        assert ok and abs(dl + (new - rho.flat[5])) <= 1e-12 * new      # no photon: l = -mu
    s.close()
