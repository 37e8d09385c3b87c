"""The partial NMO by reference curvatures far outside any physical range: the
call ends, muted outputs are zero and the transpose stays the transpose."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2505_00387_gb300 import synthetic as syn

from gpu_util import dev, gpu_plan, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_00387_gb300 import build
    build.build()


@pytest.mark.parametrize("interp", ["keys", "linear"])
@pytest.mark.parametrize("q_ref", [-1e300, -1e10, -1e8, -1.0, 1.0, 1e10, 1e300])
def test_extreme_reference_curvature(q_ref, interp):
    """r^2 / dt^2 is up to 1e11 here: every output but those of the zero-offset
    trace is muted or reads past the record."""
    g = syn.small_cube()
    hx, hy = g.hx.copy(), g.hy.copy()
    hx[7] = hy[7] = 0.0
    gp = gpu_plan(syn.Gather(g.nt, g.dt, g.ntau, g.nq, g.q0, g.dq, g.ntheta, hx, hy), interp=interp)
    d = np.random.default_rng(5).standard_normal((g.nt, g.ntr)).astype(np.float32)
    want = np.zeros_like(d)
    want[:, 7] = d[:, 7]
    for transpose in (False, True):
        out = host(gp.partial_nmo(dev(d), q_ref, transpose=transpose), d.shape)
        assert np.array_equal(out, want)
