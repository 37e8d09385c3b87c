"""Rounding of the block FFTs (plans on natural-order spectra).

Their radix networks let the compiler contract a multiplication by sqrt(1/2)
into the add that follows it.  Two-wide adds written in PTX keep it from doing
so and round the product once more: 1.7 % more error against 64 bits on
256-sample frames with the direct sum (forward 2.850e-7 against 2.801e-7,
adjoint 2.849e-7 against 2.810e-7, the same inputs).  The bound lies half way."""
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


def test_direct_plan_of_short_frames():
    nt, nq, nth = 90, 32, 8
    rng = np.random.default_rng(5)
    hx, hy = syn.disc_offsets(rng, 64, 2000.0)
    q0, dq = syn.q_axis(nq)
    g = syn.Gather(nt, 4.0 / nt, nt, nq, q0, dq, nth, hx, hy)
    kw = dict(q_axis=np.linspace(1 / 3500.0, 1 / 1500.0, nq) ** 2)
    p, gp = oracle_plan(g, **kw), gpu_plan(g, **kw)
    assert gp.info.nfft == 256
    rng = np.random.default_rng(3)
    m = rng.standard_normal((nt, nq, nth)).astype(np.float32).astype(np.float64)
    d = rng.standard_normal((nt, 64)).astype(np.float32).astype(np.float64)
    assert rel(host(gp.forward(dev(m)), d.shape), ops.forward(p, m)) < 2.826e-7
    assert rel(host(gp.adjoint(dev(d)), m.shape), ops.adjoint(p, d)) < 2.829e-7
