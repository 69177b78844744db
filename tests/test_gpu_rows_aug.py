"""The row-run form's photon-count step: blocks of nine and ten update teams on
tiles with a patch for each of them, against the general form (every chain,
count and decision the same bit for bit)."""
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
