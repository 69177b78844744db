"""Which kernel form a plan runs, as bdecon_get_form reports it.

Every form gives the same chains, so a comparison of chains says nothing about
a form that silently stopped applying.  Expected here, from the rules of the
planner: the row-run form for float problems of stride 3 and up whose window
box fits the TMA limit (PSF side 59 at three classes a run), except augmented
problems on a finer lattice or of one-patch one-team plans of one or two warps,
given block warps, staging and the lean switch."""
import numpy as np
import pytest

from paper_2411_00991_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2411_00991_gb300 import bdecon  # noqa: E402


def _sampler(p, precision=bdecon.BDECON_FP32, T=12):
    return bdecon.Sampler(p, precision=precision, max_sweeps=T)


@pytest.mark.parametrize("kw,augmented,per_team", [
    (dict(H=17, W=13, L=3), False, 1),                       # a warp per class of the row
    (dict(H=17, W=13, L=3), True, 1),
    (dict(H=16, W=19, L=5, stride=7), False, 1),
    (dict(H=41, W=60, L=17), False, 3),
    (dict(H=41, W=60, L=17), True, 3),
    (dict(H=64, W=66, L=59, sigma=9.0), False, 3),           # the widest window box
    (dict(H=64, W=66, L=61, sigma=9.0), False, 0),           # above it
    (dict(H=20, W=22, L=1, stride=2), False, 0),             # two classes a row
    (dict(H=20, W=22, L=7, subpixel=2), False, 1),
    (dict(H=20, W=22, L=7, subpixel=2), True, 0),            # augmented, finer lattice
    (dict(H=400, W=400, L=11), True, 0),                     # augmented, one patch, one team of two warps
])
def test_form_of_the_automatic_plan(kw, augmented, per_team):
    p = synth.small_problem(seed=17, **kw)
    p.augmented = augmented
    s = _sampler(p)
    f = s.form()
    assert f["per_team"] == per_team and (f["run"] > 0) == (per_team > 0)
    assert f["run"] % max(1, per_team) == 0 and f["run"] <= 16
    if kw["H"] == 400:
        assert f["one_team"] == 1
    s.close()
    if not augmented:
        s = _sampler(p, bdecon.BDECON_FP64)
        assert s.form()["run"] == 0
        s.close()


def test_settings_that_keep_the_class_by_class_forms():
    s = _sampler(synth.small_problem(H=41, W=60, L=17, seed=17))
    assert s.form()["run"] > 0 and s.form()["resident"] == 1
    s.set_plan(2, 3, 0)
    assert s.form()["run"] > 0 and s.form()["resident"] == 0
    s.set_plan(2, 3, 4)
    assert s.form()["run"] == 0
    s.set_plan(0, 0, 0)
    for mode in (0, 1):
        s.set_lean(mode)
        assert s.form()["run"] == 0
    s.set_lean(-1)
    s.set_staging(True)
    assert s.form()["run"] == 0
    s.set_staging(False)
    assert s.form()["run"] > 0
    s.close()


@pytest.mark.parametrize("warps,L,per_team", [(1, 13, 1), (2, 19, 3), (4, 25, 5), (4, 31, 4), (8, 31, 3)])
def test_every_team_width_matches_the_general_form(warps, L, per_team):
    p = synth.small_problem(H=48, W=53, L=L, sigma=2.0, seed=23, refresh_every=4)
    p.team_warps = warps
    out = []
    for lean, plan in ((0, None), (-1, None), (-1, (2, 2))):
        s = _sampler(p)
        s.set_lean(lean)
        if plan:
            s.set_plan(*plan, 0)
        assert s.form()["per_team"] == (per_team if lean else 0)
        s.sweep(6)
        out.append((s.get_state()[0], s.trace(), s.get_mu()))
        s.close()
    for o in out[1:]:
        for x, y in zip(o, out[0]):
            np.testing.assert_array_equal(x, y)


def test_one_patch_general_plan_without_room_for_the_one_team_form():
    # 512 x 512, four-warp teams, one patch a block: the lean form holds its 1024
    # blocks (8 of 128 threads an SM), the one-team form does not (80 registers: 6)
    p = synth.widefield_512()
    p.truth = None
    p.team_warps = 4
    out = []
    for plan in (None, (2, 2, 0)):
        s = _sampler(p)
        s.set_lean(1)
        if plan:
            s.set_plan(*plan)
        f, pl = s.form(), s.get_plan()
        assert f["run"] == 0 and f["one_team"] == 0 and s.lean() == 1
        if plan is None:
            assert (pl["tile_i"], pl["tile_j"], pl["warps"]) == (1, 1, 4)
        s.sweep(3)
        out.append((s.get_state()[0], s.trace(), s.get_mu()))
        s.close()
    for x, y in zip(*out):
        np.testing.assert_array_equal(x, y)
