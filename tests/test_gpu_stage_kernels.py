"""The operators' own kernels stage by stage.

aahrt_apply_stage runs the time stages of bins-fastest plans on natural-order
spectra with the shared-memory FFT kernels; under the test hook it runs the
register-FFT kernels of forward, adjoint and solves (through a transposition),
so every bin and row they produce is compared here before any other stage can
dilute an error.  Stages against the oracle: 2e-6 relative L2 for the time
stages and 1e-5 for the slice steps (the bounds of the parity tests), and no
single column further off than 1e-5 (2e-6 of the whole falls on one column of
25 at most)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ops
from paper_2505_00387_gb300 import _lib as L
from paper_2505_00387_gb300 import synthetic as syn
from paper_2505_00387_gb300.plan import AahrtPlan

from gpu_util import dev, gpu_plan, host, oracle_H, oracle_plan, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_00387_gb300 import build
    build.build()


def _gather(nt, ntau, nq, nth, ntr, seed=60):
    rng = np.random.default_rng(seed)
    hx, hy = syn.disc_offsets(rng, ntr, 1500.0)
    q0, dq = syn.q_axis(nq)
    return syn.Gather(nt, 4.0 / nt, ntau, nq, q0, dq, nth, hx, hy)


def _c64(x):
    return torch.from_numpy(np.ascontiguousarray(x, dtype=np.complex64).ravel()).cuda()


def _columns(a, b, tol):
    """Whole and worst-column relative L2 of [rows][columns] arrays."""
    a, b = a.reshape(a.shape[0], -1), b.reshape(b.shape[0], -1)
    assert rel(a, b) < tol
    err = np.linalg.norm(a - b, axis=0) / np.linalg.norm(b, axis=0)
    assert err.max() < max(1e-5, tol)


def _time_stages(gp, p, rng, nb):
    m = rng.standard_normal((p.ntau, p.nq * p.ntheta)).astype(np.float32).astype(np.float64)
    d = rng.standard_normal((p.nt, p.ntr)).astype(np.float32).astype(np.float64)
    _columns(host(gp.apply_stage(0, dev(m)), (nb, p.nq * p.ntheta)),
             ops.rfft_bins(p, ops.stretch(p, m)), 2e-6)
    _columns(host(gp.apply_stage(3, dev(d)), (nb, p.ntr)),
             ops.rfft_bins(p, ops.unstretch_T(p, d)), 2e-6)
    for stage, cols, back in ((2, p.ntr, ops.unstretch), (5, p.nq * p.ntheta, ops.stretch_T)):
        S = (rng.standard_normal((nb, cols)) + 1j * rng.standard_normal((nb, cols)))
        S = S.astype(np.complex64).astype(np.complex128)
        want = back(p, oracle_H(p, S))
        _columns(host(gp.apply_stage(stage, _c64(S)), want.shape), want, 2e-6)


@pytest.mark.parametrize("nt,ntau,nfft,interp", [
    (200, 200, 512, "keys"), (400, 300, 1024, "linear"), (800, 900, 2048, "keys"),
    (1600, 1600, 4096, "keys"), (3200, 3200, 8192, "linear")])
def test_time_stages(nt, ntau, nfft, interp):
    """Odd column counts on both sides, both kinds of kernels."""
    g = _gather(nt, ntau, 17, 3, 23)
    p, gp = oracle_plan(g, interp=interp), gpu_plan(g, interp=interp)
    assert gp.info.nfft == nfft
    rng = np.random.default_rng(61)
    _time_stages(gp, p, rng, p.nbins)
    L.aahrt_plan_test_stage_frames(gp.handle, True)
    _time_stages(gp, p, rng, p.nbins)


def test_slice_stages_of_uneven_cubes():
    gs = [_gather(300, 300, 33, 5, n, seed=62 + n) for n in (41, 3, 70)]
    gp = AahrtPlan.batched(gs)
    r2max = max(float(np.max(g.hx ** 2 + g.hy ** 2)) for g in gs)
    os_ = [oracle_plan(g, r2max=r2max) for g in gs]
    rng = np.random.default_rng(63)
    nb = os_[0].nbins
    cplx = lambda *s: (rng.standard_normal(s) + 1j * rng.standard_normal(s)).astype(np.complex64)
    X = [cplx(nb, 33, 5) for _ in gs]
    Y = [cplx(nb, g.ntr) for g in gs]
    Yg = host(gp.apply_stage(1, _c64(np.concatenate([x.ravel() for x in X]))))
    Xg = host(gp.apply_stage(4, _c64(np.concatenate([y.ravel() for y in Y]))))
    for c, (g, p) in enumerate(zip(gs, os_)):
        o = nb * sum(x.ntr for x in gs[:c])
        yo = ops.slice_forward(p, X[c].astype(np.complex128)) / p.nfft
        assert rel(Yg[o:o + nb * g.ntr].reshape(yo.shape), yo) < 1e-5
        xo = ops.slice_adjoint(p, Y[c].astype(np.complex128)) / p.nfft
        assert rel(Xg[c * nb * 165:(c + 1) * nb * 165].reshape(xo.shape), xo) < 1e-5


def test_hook_refuses_plans_on_natural_spectra():
    g = _gather(200, 200, 17, 3, 23)
    gp = gpu_plan(g, slice_interp="direct")
    with pytest.raises(L.AahrtError):
        L.aahrt_plan_test_stage_frames(gp.handle, True)


def _time(fn, n=10):
    best = 1e30
    for _ in range(5):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        for _ in range(n):
            fn()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) / n)
    return best


def test_time_of_the_adjoint_slice_stage():
    """One slice step with its spectra moved between the layouts takes less than
    the whole adjoint (it took 1.15 times as long when the bound was a pass over
    the spectrum for every azimuth group)."""
    g = _gather(1001, 1001, 100, 36, 2000)
    gp = gpu_plan(g)
    d = torch.randn(gp.data_len, device="cuda")
    Y = gp.apply_stage(3, d)
    X = gp.apply_stage(4, Y)
    assert _time(lambda: gp.apply_stage(4, Y, X)) < 0.9 * _time(lambda: gp.adjoint(d))
