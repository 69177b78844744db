"""Double chains do not depend on how much device memory there is: with the
likelihood records in the workspace, in page-locked host memory because the
workspace is short, or in a server whose budget is, the results are the same
bit for bit."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2411_00991_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2411_00991_gb300 import bdecon  # noqa: E402

FP64 = bdecon.BDECON_FP64


def _sizes(probs, T, flags=0):
    """Workspace bytes with the records and without them."""
    full = bdecon.Sampler.workspace_size(probs, precision=FP64, max_sweeps=T, flags=flags)
    rec = [112 * p.H * ((p.W + 3) // 4 * 4) for p in probs]
    return full, full - sum((r + 255) // 256 * 256 * p.n_chains for r, p in zip(rec, probs) if not p.augmented)


def _run(probs, T, nbytes, flags=bdecon.FLAG_ACCEPT_LOG, setup=None):
    buf = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    s = bdecon.Sampler(probs, precision=FP64, max_sweeps=T, flags=flags, workspace=(buf.data_ptr(), nbytes))
    where = s.records()
    if setup:
        setup(s)
    s.sweep(T - 3)
    s.sweep(3)
    out = []
    for p, q in enumerate(probs):
        for c in range(q.n_chains):
            out += [s.get_state(p, c)[0], s.trace(p, c), s.get_mu(p, c), s.accept_log(p, c)]
        if not q.augmented:
            out.append(np.array([s.delta(m, float(out[0].flat[0]), p) for m in (0, 7)]))
        out.append(s.posterior_mean(p))
    s.close()
    return where, out


CASES = [
    [dict(H=20, W=24, L=5)],
    [dict(H=41, W=37, L=9, maps=True, n_chains=2)],
    [dict(H=50, W=43, L=17, sigma=1.3, peak=200.0, burn_in=4)],
    [dict(H=20, W=22, L=7, subpixel=2)],
    [dict(H=20, W=24, L=5), dict(H=30, W=21, L=9, n_chains=2), dict(H=18, W=18, L=5)],   # a batch, the last augmented
]


@pytest.mark.parametrize("kws", CASES, ids=lambda k: "+".join("%dx%dL%d" % (q["H"], q["W"], q["L"]) for q in k))
def test_chains_with_records_in_host_memory(kws):
    probs = [synth.small_problem(seed=41 + k, **dict(dict(refresh_every=5), **kw)) for k, kw in enumerate(kws)]
    if len(probs) > 1:
        probs[-1].augmented = True
    T = 13
    full, short = _sizes(probs, T, bdecon.FLAG_ACCEPT_LOG)
    where, want = _run(probs, T, full)
    assert where == 1
    for nbytes, setup in ((short, None), (full - 256, None), (short, lambda s: s.set_graph(True)),
                          (short, lambda s: s.autotune(2))):
        where, got = _run(probs, T, nbytes, setup=setup)
        assert where == 2
        for x, y in zip(got, want):
            np.testing.assert_array_equal(x, y)
    with pytest.raises(bdecon.BdeconError) as ei:
        _run(probs, T, short - 1)
    assert ei.value.status == 2
    bdecon.set_tuning_cache(True)


def test_host_records_chain_equals_the_oracle():
    p = synth.small_problem(H=20, W=24, L=5, seed=44, refresh_every=6)
    T = 15
    where, got = _run([p], T, _sizes([p], T, bdecon.FLAG_ACCEPT_LOG)[1])
    assert where == 2
    ref = O.Oracle(p).run(T, want_acc_log=True)
    np.testing.assert_array_equal(got[3], ref["acc_log"])
    np.testing.assert_allclose(got[0], ref["rho"], rtol=1e-12)
    np.testing.assert_allclose(got[1], ref["trace"], rtol=1e-12)


def test_records_of_other_samplers():
    p = synth.small_problem(H=20, W=24, L=5, seed=45)
    for precision, augmented, where in ((bdecon.BDECON_FP32, False, 0), (FP64, True, 0), (FP64, False, 1)):
        p.augmented = augmented
        s = bdecon.Sampler(p, precision=precision, max_sweeps=4)
        assert s.records() == where
        s.close()


@pytest.mark.parametrize("room", ["all", "no records"])
def test_server_job_equals_the_job_alone(room):
    p = synth.small_problem(H=60, W=52, L=9, seed=46, refresh_every=6)
    T = 14
    s = bdecon.Sampler(p, precision=FP64, max_sweeps=T)
    s.sweep(T)
    want = s.posterior_mean()
    s.close()
    full, short = _sizes([p], T)
    srv = bdecon.Server(mem_budget=full if room == "all" else short, max_jobs=2, segment_sweeps=4, precision=FP64)
    ids = [srv.submit(p, T) for _ in range(2)]
    for i in ids:
        np.testing.assert_array_equal(srv.result(i)[0], want)
    srv.close()
    srv = bdecon.Server(mem_budget=short - 1, max_jobs=2, segment_sweeps=4, precision=FP64)
    with pytest.raises(bdecon.BdeconError):
        srv.result(srv.submit(p, T))
    srv.close()
