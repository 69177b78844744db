"""Window tensor maps rewritten in place: plans changed on a live handle, and
handles created one after another at the same device addresses, give the chains
of the class-by-class form, whose windows no tensor map describes."""
import numpy as np
import pytest

from paper_2411_00991_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2411_00991_gb300 import bdecon  # noqa: E402


def _state(s, n):
    return [x for p in range(n) for x in (s.get_state(p)[0], s.trace(p), s.get_mu(p))]


def test_maps_of_changing_plans():
    probs = [synth.small_problem(H=40, W=53, L=9, seed=71, refresh_every=7),
             synth.small_problem(H=33, W=20, L=9, seed=72, refresh_every=7, n_chains=2),
             synth.small_problem(H=50, W=47, L=17, sigma=1.5, seed=73, refresh_every=7)]
    T, n = 24, len(probs)
    ref = bdecon.Sampler(probs, max_sweeps=T)
    ref.set_lean(0)
    ref.sweep(T)
    s = bdecon.Sampler(probs, max_sweeps=T)
    for k in range(T // 4):
        s.sweep(2)
        s.set_plan(1 + k % 3, 2, 0, k % n)       # other tiles
        s.sweep(1)
        s.set_grouping(k % 2 == 0)               # other chains in a launch
        s.set_staging(k % 3 == 0)
        s.sweep(1)
    for x, y in zip(_state(s, n), _state(ref, n)):
        np.testing.assert_array_equal(x, y)
    s.close()
    ref.close()


def test_maps_at_reused_addresses():
    rng = np.random.default_rng(5)
    for k in range(12):
        L = int(rng.choice([5, 9, 13, 17]))
        kw = dict(H=int(rng.integers(20, 70)), W=int(rng.integers(20, 70)), L=L, sigma=1.5, seed=80 + k)
        out = []
        nbytes = None
        for lean in (-1, 0):
            p = synth.small_problem(**kw)
            if nbytes is None:
                nbytes = bdecon.Sampler.workspace_size(p, max_sweeps=8)
            s = bdecon.Sampler(p, max_sweeps=8, workspace=(_buffer().data_ptr(), nbytes))
            s.set_lean(lean)
            s.sweep(4)
            out.append(_state(s, 1))
            s.close()
        for x, y in zip(*out):
            np.testing.assert_array_equal(x, y)


_BUF = []


def _buffer():
    if not _BUF:   # one device buffer for every handle: the maps land at addresses used before
        _BUF.append(torch.zeros(64 << 20, dtype=torch.uint8, device="cuda"))
    return _BUF[0]
