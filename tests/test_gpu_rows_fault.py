"""Waits that run out in the row-run form: a block that never publishes makes
its neighbours give up (a bounded wait, no GPU fault).  On frames lower or
narrower than the window most cells of a window lie outside the frame, and a
block that gave up has no window of its own run; it must read none of their data.
The host reads the timeout, and the next handle samples as usual."""
import numpy as np
import pytest

from paper_2411_00991_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2411_00991_gb300 import bdecon  # noqa: E402


@pytest.mark.parametrize("kw,augmented", [
    (dict(H=1, W=60, L=9), False),
    (dict(H=60, W=1, L=9), False),
    (dict(H=2, W=70, L=17, peak=300.0), False),
    (dict(H=41, W=60, L=17, peak=300.0), False),
    (dict(H=1, W=60, L=9), True),
    (dict(H=8, W=30, L=7, subpixel=2), False),
])
def test_timeout_on_frames_below_the_window(kw, augmented):
    p = synth.small_problem(seed=61, refresh_every=0, **kw)
    p.augmented = augmented
    s = bdecon.Sampler(p, precision=bdecon.BDECON_FP32, max_sweeps=8)
    assert s.form()["run"] > 0
    s.sweep(1)
    s.set_fault(s.get_plan()["blocks"] // 2, 50_000_000)
    s.sweep(3)
    with pytest.raises(bdecon.BdeconError) as ei:
        s.sync()
    assert ei.value.status == 4
    s.close()
    out = []
    for lean in (0, -1):
        s = bdecon.Sampler(p, precision=bdecon.BDECON_FP32, max_sweeps=8)
        s.set_lean(lean)
        s.sweep(4)
        out.append((s.get_state()[0], s.trace()))
        s.close()
    for x, y in zip(*out):
        np.testing.assert_array_equal(x, y)
