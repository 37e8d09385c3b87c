"""Time of the partial NMO's transpose beside the plan's adjoint.

The transpose is one light pass over the data: on a small cube it stays below
1.5 times the adjoint, whose stack it precedes in an inversion (a thread that
walks several rows one after another took 3.4 adjoints there)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2505_00387_gb300 import synthetic as syn

from gpu_util import dev, gpu_plan

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_00387_gb300 import build
    build.build()


def _time(fn, n=20):
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


def test_transposed_partial_nmo_on_a_small_cube():
    g = syn.small_cube()
    gp = gpu_plan(g)
    d = dev(np.random.default_rng(3).standard_normal((g.nt, g.ntr)))
    assert (_time(lambda: gp.partial_nmo(d, 1e-7, transpose=True)) <
            1.5 * _time(lambda: gp.adjoint(d)))
