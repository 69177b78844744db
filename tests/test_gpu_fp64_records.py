"""Double chains' cumulant records against the exact photon sums.

The double sweep evaluates a likelihood change from each camera pixel's
cumulant record (series up to |log mu'/mu| of about a tenth, the exact sum
beyond), and moves the record with accepted updates.  A likelihood change is
compared with 40-digit sums of Eq. 6 on a one-pixel PSF, at sizes on both
sides of the series' two limits, with fresh records and with records moved by
many accepted updates.  Tolerance: the change is a difference of terms of the
size of |mu' - mu|, so a few units in the last place of that."""
import math

import numpy as np
import pytest

from paper_2411_00991_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
mp = pytest.importorskip("mpmath")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2411_00991_gb300 import bdecon  # noqa: E402


def _exact(g, w, v, m, mn):
    with mp.workdps(40):
        c, is2 = (mp.mpf(float(w)) - 100) / mp.mpf(g), mp.mpf(g) ** 2 / mp.mpf(float(v))

        def log_sum(x):
            lo, hi = max(0, int(x - 14 * math.sqrt(x) - 25)), int(max(x, float(c)) + 14 * math.sqrt(max(x, 1.0)) + 40)
            lt = [-(c - f) ** 2 * is2 / 2 + f * mp.log(x) - mp.loggamma(f + 1) for f in range(lo, hi)]
            top = max(lt)
            return top + mp.log(mp.fsum(mp.exp(y - top) for y in lt))
        return log_sum(mp.mpf(mn)) - log_sum(mp.mpf(m)) - (mp.mpf(mn) - mp.mpf(m))


@pytest.mark.parametrize("sweeps", [0, 200])
def test_likelihood_change_from_records(sweeps):
    rng = np.random.default_rng(8)
    n, g = 12, 2.1
    mu = np.exp(rng.uniform(math.log(0.3), math.log(300.0), (n, n)))
    var = rng.gamma(2.0, 1.0, (n, n)).astype(np.float32) + np.float32(0.05)
    img = (g * rng.poisson(mu) + 100 + rng.normal(size=(n, n)) * np.sqrt(var)).astype(np.float32)
    p = synth.Problem(image=img, psf=np.ones((1, 1)), gain=g, offset=100.0, var=var, stride=1, seed=1, refresh_every=0)
    s = bdecon.Sampler(p, precision=bdecon.BDECON_FP64, max_sweeps=400)
    s.set_state(mu, 0)
    if sweeps:
        s.sweep(sweeps)
        assert s.accept_counts().sum() > 50 * n * n          # every record was moved many times
        mu = s.get_state()[0]
    for d in (1e-9, 0.99e-3, 1.01e-3, 0.05, 0.119, 0.121, 0.5):
        for sign in (-1, 1):
            for i in rng.integers(0, n * n, 6):
                m = float(mu.flat[i])
                new = m * (1 + sign * d)
                ok, dl, _ = s.delta(int(i), new)
                ref = _exact(g, img.flat[i], var.flat[i], m, new)
                assert ok and abs(float(mp.mpf(dl) - ref)) <= 4e-15 * abs(new - m), (d, sign, m)
    s.close()
