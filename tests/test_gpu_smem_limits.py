"""Set-up and refresh of every patch side around the default shared-memory limit
(48 KB with the kernels' static arrays), smallest first: none relies on a limit
that an earlier, larger problem raised."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

PROGRAM = """
from oracle import oracle as O
from paper_2411_00991_gb300 import bdecon, synth
for L in (43, 45, 47):
    for precision in (bdecon.BDECON_FP64, bdecon.BDECON_FP32):
        p = synth.small_problem(H=12, W=10, L=L, sigma=3.0, seed=L)
        s = bdecon.Sampler(p, precision=precision, max_sweeps=4)
        ref = O.Oracle(p).log_posterior(s.get_state()[0])
        assert abs(s.log_posterior() - ref) <= 1e-12 * abs(ref), (L, precision)
        s.close()
"""


def test_patch_sides_around_the_default_limit():
    # (a process of its own: limits last as long as the process)
    subprocess.run([sys.executable, "-c", PROGRAM], check=True)
