"""The row-run form of the float sweep kernel against the general form.

It scores runs of classes at once and reads its windows through the TMA
engine; every cell, entry and sum is taken by the same thread in the same
order, so chains -- objects, expected images, traces, accept decisions, kept
objects -- are bit-identical to the general form's (lean mode 0), on one-patch
and multi-patch tiles, ragged frames, strides above the PSF side, and at the
ends of its range (three classes a row; window boxes above the TMA limit,
which keep the general form)."""
import numpy as np
import pytest

from paper_2411_00991_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2411_00991_gb300 import bdecon  # noqa: E402


def _run(p, T, lean, plan):
    s = bdecon.Sampler(p, precision=bdecon.BDECON_FP32, max_sweeps=T + 4, flags=bdecon.FLAG_ACCEPT_LOG | bdecon.FLAG_SECOND_MOMENT)
    if lean is not None:
        s.set_lean(lean)
    if plan is not None:
        s.set_plan(plan[0], plan[1], 0)
    s.sweep(T - 3)
    s.sweep(3)
    out = []
    for c in range(p.n_chains):
        rho, t = s.get_state(0, c)
        tr = s.trace(0, c)
        assert t == T and np.isfinite(tr).all()
        out += [rho, tr, s.get_mu(0, c), s.accept_counts(0, c), s.accept_log(0, c), s.get_steps(0, c), s.samples(0, c)]
        if p.augmented:
            out.append(s.get_phi(0, c))
    out += [s.posterior_mean(), s.posterior_std()]
    s.close()
    return out


CASES = [
    dict(H=17, W=13, L=3, maps=True, n_chains=2),           # three classes a row, one ragged patch row
    dict(H=20, W=24, L=5),                                  # ragged on both sides
    dict(H=16, W=19, L=5, stride=7),                        # stride above the PSF side
    dict(H=5, W=40, L=9),                                   # one row of patches, frame below the window
    dict(H=26, W=22, L=11, sigma=1.8, peak=300.0),          # large changes: the exact sums
    dict(H=41, W=60, L=17, sigma=1.3, maps=True),           # three-warp teams
    dict(H=70, W=65, L=31, sigma=4.0, peak=5.0),            # eight-warp teams
    dict(H=60, W=47, L=55, sigma=8.0),                      # the widest window box
    dict(H=64, W=66, L=59, sigma=9.0),                      # above it: the general form
    dict(H=20, W=22, L=7, subpixel=2),                      # finer lattices: every phase of the kernel
    dict(H=15, W=17, L=5, subpixel=3, stride=9, maps=True),
    dict(H=40, W=33, L=25, sigma=5.0, subpixel=2, n_chains=2),
]


@pytest.mark.parametrize("kw", CASES, ids=lambda kw: "%dx%dL%df%d" % (kw["H"], kw["W"], kw["L"], kw.get("subpixel", 1)))
@pytest.mark.parametrize("augmented", [False, True])
def test_rows_are_bit_identical_to_the_general_form(kw, augmented):
    p = synth.small_problem(seed=17, refresh_every=4, burn_in=2, **kw)
    p.augmented, p.n_samples, p.sample_every = augmented, 2, 2
    T = 8
    want = _run(p, T, 0, None)
    for plan in (None, (2, 3), (1, 4)):
        for x, y in zip(_run(p, T, None, plan), want):
            np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("warps,L", [(1, 13), (2, 19), (4, 25), (6, 21)])
def test_rows_with_given_teams_and_adaptation(warps, L):
    # teams of every block shape (VG 1, 3, 4 and 5 classes a team), adapting scales
    p = synth.small_problem(H=48, W=53, L=L, sigma=2.0, seed=23, refresh_every=0, burn_in=5)
    p.team_warps, p.adapt_target, p.n_samples = warps, 0.2, 1
    want = _run(p, 9, 0, None)
    for plan in (None, (2, 2)):
        for x, y in zip(_run(p, 9, None, plan), want):
            np.testing.assert_array_equal(x, y)
