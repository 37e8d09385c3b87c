"""The bins-fastest slice kernels at the edges of their range, against the
FP64 oracle: every q grid size they serve (32 to 512 points) and its
neighbours outside (16, 1024: the bin-per-block kernels), odd bin counts (a
part tile), one to three azimuths, given groups, empty azimuth intervals,
uneven folds.  Tolerances: the operator bound of the parity tests (1e-4
relative L2; 5e-4 for five taps)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ops
from paper_2505_00387_gb300 import synthetic as syn

from gpu_util import dev, gpu_plan, host, oracle_plan, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_00387_gb300 import build
    build.build()


def _gather(nq, nth, ntr=60, nt=90, sector=np.pi, seed=70):
    rng = np.random.default_rng(seed)
    hx, hy = syn.disc_offsets(rng, ntr, 1200.0, 0.3, sector)
    q0, dq = syn.q_axis(nq)
    return syn.Gather(nt, 0.012, nt, nq, q0, dq, nth, hx, hy)


def _check(g, tol, p_kw=None, **kw):
    p = oracle_plan(g, **(p_kw or {}))
    gp = gpu_plan(g, **kw)
    rng = np.random.default_rng(71)
    m = rng.standard_normal((g.ntau, g.nq, g.ntheta))
    d = rng.standard_normal((g.nt, g.ntr))
    assert rel(host(gp.forward(dev(m)), (g.nt, g.ntr)), ops.forward(p, m)) < tol
    assert rel(host(gp.adjoint(dev(d)), m.shape), ops.adjoint(p, d)) < tol
    return gp, m, d


@pytest.mark.parametrize("nq,nos", [(8, 16), (9, 32), (16, 32), (17, 64), (33, 128), (64, 128),
                                    (100, 256), (129, 512), (256, 512), (257, 1024)])
def test_grid_sizes(nq, nos):
    gp, _, _ = _check(_gather(nq, 4), 1e-4)
    assert gp.info.nq_os == nos


@pytest.mark.parametrize("w", [5, 12])
@pytest.mark.parametrize("nq", [30, 60, 120, 200])
def test_widths(nq, w):
    _check(_gather(nq, 3), 5e-4 if w < 6 else 1e-4, spread_width=w)


@pytest.mark.parametrize("nth,tg", [(1, 0), (2, 0), (2, 1), (3, 2), (7, 3)])
def test_azimuth_groups(nth, tg):
    _check(_gather(40, nth), 1e-4, theta_group=tg)


def test_part_tile_and_dense_axis():
    """A bin count that is no multiple of the tile, and a q grid under 2 nq."""
    g = _gather(40, 3)
    gp, _, _ = _check(g, 1e-4, p_kw=dict(fmax=30.0), fmax=30.0)
    assert gp.info.nbins % 16
    _check(_gather(50, 3), 1e-4, sigma_q=1.25, spread_width=12)


def test_empty_intervals():
    """A 40-degree sector of 12 azimuths: most slices see no trace, and their
    adjoint spectrum is exactly zero (the synthesis packs two columns into one
    complex FFT, so the model only is to rounding)."""
    g = _gather(40, 12, sector=np.deg2rad(40.0))
    gp, _, d = _check(g, 1e-4)
    X = host(gp.apply_stage(4, gp.apply_stage(3, dev(d))), (gp.info.nbins, g.nq, g.ntheta))
    p = oracle_plan(g)
    used = set(p.j0[p.w0 > 0]) | set(p.j1[p.w1 > 0])
    assert len(used) < 6
    for j in set(range(12)) - used:
        assert not X[:, :, j].any()


def test_stages_compose():
    """The stages on natural-order spectra (X[bin][q][theta], Y[bin][trace])
    compose to the operators computed in the plan's own layout, on a batch of
    uneven folds (FP32 rounding of identical sums: 1e-6)."""
    from paper_2505_00387_gb300.plan import AahrtPlan
    gs = [_gather(40, 5, ntr=n, seed=80 + n) for n in (37, 5, 64)]
    gp = AahrtPlan.batched(gs)
    rng = np.random.default_rng(72)
    m = dev(rng.standard_normal(gp.model_len))
    d = dev(rng.standard_normal(gp.data_len))
    f = gp.apply_stage(2, gp.apply_stage(1, gp.apply_stage(0, m)))
    a = gp.apply_stage(5, gp.apply_stage(4, gp.apply_stage(3, d)))
    assert rel(host(f), host(gp.forward(m))) < 1e-6
    assert rel(host(a), host(gp.adjoint(d))) < 1e-6
