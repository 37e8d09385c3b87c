"""The register-FFT time kernels over every frame length they serve (512 to
8192 samples) and the lengths beside it (256, 16384), with odd column counts,
a model axis shorter and longer than the data's, linear interpolation and an
odd number of bins: operators (1e-4 relative L2 against the FP64 oracle) and
two fused FISTA iterations (1e-3), the bounds of the parity tests."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import fista, ops
from paper_2505_00387_gb300 import synthetic as syn

from gpu_util import dev, gpu_plan, host, oracle_plan, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_00387_gb300 import build
    build.build()


def _run(nt, ntau, interp, ntr=7, nq=17, nth=3, fmax=0.0):
    rng = np.random.default_rng(90)
    dt = 4.0 / nt
    hx, hy = syn.disc_offsets(rng, ntr, 1500.0)
    q0, dq = syn.q_axis(nq)
    g = syn.Gather(nt, dt, ntau, nq, q0, dq, nth, hx, hy)
    kw = dict(interp=interp, fmax=fmax)
    p, gp = oracle_plan(g, **kw), gpu_plan(g, **kw)
    m = rng.standard_normal((ntau, nq, nth))
    d = rng.standard_normal((nt, ntr))
    assert rel(host(gp.forward(dev(m)), d.shape), ops.forward(p, m)) < 1e-4
    adj = ops.adjoint(p, d)
    assert rel(host(gp.adjoint(dev(d)), m.shape), adj) < 1e-4
    lam = 0.05 * float(np.abs(adj).max())
    gamma = 0.5 / fista.power_sigma2(p, d, iters=5)
    ms, _ = gp.sparse_solve(dev(d), lam, 2, gamma=gamma)
    assert rel(host(ms, m.shape), fista.solve(p, d, lam, 2, gamma)) < 1e-3
    return gp


@pytest.mark.parametrize("nt,nfft", [(100, 256), (200, 512), (400, 1024), (800, 2048),
                                     (1600, 4096), (3200, 8192), (6400, 16384)])
def test_frame_lengths(nt, nfft):
    gp = _run(nt, nt, "keys")
    assert gp.info.nfft == nfft


@pytest.mark.parametrize("nt,ntau,interp,ntr", [(300, 90, "keys", 1), (300, 411, "linear", 2),
                                                (1001, 40, "linear", 5), (1001, 1100, "keys", 6)])
def test_axes(nt, ntau, interp, ntr):
    _run(nt, ntau, interp, ntr=ntr, nth=2)


def test_odd_bins():
    """Adjacent bin counts, one of them odd: its spectra's columns are 8-byte
    aligned only."""
    bins = {_run(500, 500, "keys", fmax=f).info.nbins % 2 for f in (20.0, 20.06)}
    assert bins == {0, 1}


@pytest.mark.parametrize("nt,nfft", [(200, 512), (400, 1024), (800, 2048), (1600, 4096),
                                     (3200, 8192), (6400, 16384)])
@pytest.mark.parametrize("ng,interp", [(5, "keys"), (6, "linear"), (8, "keys")])
def test_gathers_fastest(nt, nfft, ng, interp):
    """The same stages with the gathers fastest (512 to 8192 samples, and the
    length beyond), for gathers in whole 32-byte sectors, whole 16-byte pairs
    and neither: every gather of a tensor-core plan against the oracle (1e-4)."""
    rng = np.random.default_rng(91)
    hx, hy = syn.disc_offsets(rng, 9, 1500.0)
    q0, dq = syn.q_axis(17)
    g = syn.Gather(nt, 4.0 / nt, nt + 3, 17, q0, dq, 3, hx, hy)
    p = oracle_plan(g, interp=interp)
    gp = gpu_plan(g, interp=interp, ngather=ng, precision="split_bf16")
    assert gp.info.nfft == nfft
    m = rng.standard_normal((g.ntau, g.nq, g.ntheta, ng))
    d = rng.standard_normal((nt, 9, ng))
    df = host(gp.forward(dev(m)), d.shape)
    ma = host(gp.adjoint(dev(d)), m.shape)
    for i in (0, ng - 1):
        assert rel(df[..., i], ops.forward(p, m[..., i])) < 1e-4
        assert rel(ma[..., i], ops.adjoint(p, d[..., i])) < 1e-4
