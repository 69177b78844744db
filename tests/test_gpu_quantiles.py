"""Quantile maps from the warp-sort kernel: every register width and its edges
(1, 32, 33, 64, 65, 128, 129, 256 kept values a pixel, and 257, which takes the
block form), ragged pixel blocks, crops, one and several chains, both sample
types, against numpy on the same kept objects."""
import numpy as np
import pytest

from paper_2411_00991_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2411_00991_gb300 import bdecon  # noqa: E402


@pytest.mark.parametrize("precision", [bdecon.BDECON_FP32, bdecon.BDECON_FP64])
@pytest.mark.parametrize("n,chains", [(1, 1), (32, 1), (11, 3), (64, 1), (65, 1), (64, 2), (129, 1), (256, 1), (257, 1)])
def test_quantiles_match_numpy(n, chains, precision):
    p = synth.small_problem(H=11, W=9, L=3, seed=31, n_chains=chains, refresh_every=0)
    p.n_samples, p.sample_every = n, 1
    s = bdecon.Sampler(p, precision=precision, max_sweeps=n)
    s.sweep(n)
    kept = np.concatenate([s.samples(0, c) for c in range(chains)])
    assert kept.shape[0] == n * chains
    q = [0.0, 0.05, 0.5, 0.77, 1.0]
    want = np.quantile(kept, q, axis=0)
    np.testing.assert_allclose(s.posterior_quantiles(q), want, rtol=1e-15)
    np.testing.assert_allclose(s.posterior_quantiles(q, crop=True), want[:, 1:-1, 1:-1], rtol=1e-15)
    s.close()
