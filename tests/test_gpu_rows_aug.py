"""The row-run form's photon-count step against the general form (every chain,
count and decision the same bit for bit): blocks of nine and ten update teams on
tiles with a patch for each of them, and one tile over the whole frame, whose
window copies no neighbour's change orders after the block's own counts."""
import numpy as np
import pytest

from paper_2411_00991_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2411_00991_gb300 import bdecon  # noqa: E402


def _chain(p, lean, plan, T, run=None):
    s = bdecon.Sampler(p, precision=bdecon.BDECON_FP32, max_sweeps=T, flags=bdecon.FLAG_ACCEPT_LOG)
    s.set_lean(lean)
    if plan:
        s.set_plan(*plan, 0)
    if run is not None:
        assert s.form()["run"] == run
    s.sweep(T - 2)
    s.sweep(2)
    out = [s.get_state()[0], s.trace(), s.get_mu(), s.get_phi(), s.accept_log()]
    s.close()
    return out


@pytest.mark.parametrize("H,W,L,plan,run", [
    (40, 40, 9, (3, 3), 9),       # nine teams, nine patches
    (40, 40, 9, (4, 3), 9),
    (30, 60, 11, (2, 5), 10),     # ten teams, ten patches
    (60, 58, 13, (4, 4), 10),     # ten teams, sixteen patches: two rounds
])
def test_count_step_of_wide_blocks(H, W, L, plan, run):
    p = synth.small_problem(H=H, W=W, L=L, sigma=1.5, seed=31, refresh_every=5)
    p.augmented, p.team_warps = True, 1
    T = 9
    want = _chain(p, 0, None, T)
    for x, y in zip(_chain(p, -1, plan, T, run), want):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("kw,plan", [
    (dict(H=40, W=40, L=9), (6, 6)),
    (dict(H=14, W=12, L=5, sigma=1.0), (4, 4)),
    (dict(H=6, W=6, L=5, sigma=1.0, stride=11), None),    # one patch: stride above the object side
    (dict(H=41, W=60, L=17, sigma=1.3), (4, 5)),
])
def test_count_step_of_a_frame_in_one_tile(kw, plan):
    p = synth.small_problem(seed=32, refresh_every=0, **kw)
    p.augmented = True
    T = 60
    s = bdecon.Sampler(p, precision=bdecon.BDECON_FP32, max_sweeps=4)
    if plan:
        s.set_plan(*plan, 0)
    assert s.form()["run"] > 0 and s.get_plan()["blocks"] == 1
    s.close()
    want = _chain(p, 0, None, T)
    for x, y in zip(_chain(p, -1, plan, T), want):
        np.testing.assert_array_equal(x, y)
