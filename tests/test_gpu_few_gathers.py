"""Tensor-core plans where a warp of operand producers has nothing to do: row
tiles and curvature axes that do not fill the 128 rows of an A operand (the
warps past their end write nothing), gather counts below 64 (the warps past the
last gather load no B operand) and the 57-64 where every producer has its share.
Every gather is compared with the FP64 oracle (1e-4 relative L2, the bound of
the tensor-core parity tests), and a solve's residual with the oracle's
(1e-3)."""
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


def _case(ng, nq, ntr, nth=3, nt=80):
    rng = np.random.default_rng(95)
    hx, hy = syn.disc_offsets(rng, ntr, 1500.0)
    q0, dq = syn.q_axis(nq)
    g = syn.Gather(nt, 4.0 / nt, nt, nq, q0, dq, nth, hx, hy)
    gp = gpu_plan(g, ngather=ng, precision="split_bf16")
    m = rng.standard_normal((nt, nq, nth, ng))
    d = rng.standard_normal((nt, ntr, ng))
    return g, oracle_plan(g), gp, m, d


@pytest.mark.parametrize("ng,nq,ntr", [
    (1, 3, 2),          # one warp of rows
    (4, 8, 24),         # whole warps only
    (7, 20, 150),       # 50 traces a slice
    (8, 33, 385),       # a second q chunk of one sample, a second row tile
    (31, 64, 40),
    (56, 128, 40),      # a full M tile; the last gather count with idle warps
    (57, 129, 40),      # a second M tile of one row; every producer busy
    (64, 20, 150),
])
def test_every_gather(ng, nq, ntr):
    g, p, gp, m, d = _case(ng, nq, ntr)
    df = host(gp.forward(dev(m)), d.shape)
    ma = host(gp.adjoint(dev(d)), m.shape)
    gp.status()
    for i in range(ng):
        assert rel(df[..., i], ops.forward(p, m[..., i])) < 1e-4
        assert rel(ma[..., i], ops.adjoint(p, d[..., i])) < 1e-4


@pytest.mark.parametrize("ng", [5, 6, 8])
def test_all_gathers_of_a_register_fft_block(ng):
    """2048-sample frames: two pairs of gathers to a block, with a gather left
    over, a pair left over and none; a solve's residual norm is summed by the
    residual epilogue of those kernels."""
    g, p, gp, m, d = _case(ng, 17, 9, nt=800)
    df = host(gp.forward(dev(m)), d.shape)
    ma = host(gp.adjoint(dev(d)), m.shape)
    ss, iters, lam, gamma = 0.0, 2, 0.5, 1e-3
    for i in range(ng):
        assert rel(df[..., i], ops.forward(p, m[..., i])) < 1e-4
        assert rel(ma[..., i], ops.adjoint(p, d[..., i])) < 1e-4
        mi = fista.solve(p, d[..., i], lam, iters, gamma)
        ss += float(np.sum((d[..., i] - ops.forward(p, mi)) ** 2))
    _, info = gp.sparse_solve(dev(d), lam, iters, gamma=gamma)
    assert abs(info.resid_norm - np.sqrt(ss)) < 1e-3 * np.sqrt(ss)
