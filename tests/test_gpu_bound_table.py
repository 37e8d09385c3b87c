"""The spectrum bound table of bins-fastest plans between calls.

The data-side analysis raises it, the slice adjoint that reads it clears it.
An adjoint must not depend on what ran before it on the plan: amplitudes a
million times larger, the single stages, the allocation-free forward, or a call
that failed between the two kernels.  The integer spread makes the adjoint
repeatable bit for bit, so every comparison is exact."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2505_00387_gb300 import _lib as L
from paper_2505_00387_gb300 import synthetic as syn

from gpu_util import dev, gpu_plan

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_00387_gb300 import build
    build.build()


@pytest.fixture()
def case():
    g = syn.small_cube()
    rng = np.random.default_rng(41)
    d = dev(rng.standard_normal((g.nt, g.ntr)))
    m = dev(rng.standard_normal((g.ntau, g.nq, g.ntheta)))
    return gpu_plan(g), m, d, gpu_plan(g).adjoint(d)      # the last by a fresh plan


def _fail_adjoint(gp, call):
    L.aahrt_plan_test_fail_adjoint(gp.handle, True)
    with pytest.raises(L.AahrtError):
        call()
    L.aahrt_plan_test_fail_adjoint(gp.handle, False)


def test_large_then_small(case):
    gp, _, d, want = case
    gp.adjoint(1e6 * d)
    assert torch.equal(gp.adjoint(d), want)


def test_between_stages_and_the_allocation_free_forward(case):
    gp, m, d, want = case
    Y = gp.apply_stage(3, 1e6 * d)
    gp.apply_stage(4, Y)
    assert torch.equal(gp.adjoint(d), want)
    out = torch.empty(gp.data_len, device="cuda")
    L.aahrt_forward_noalloc(gp.handle, m.data_ptr(), out.data_ptr(),
                            torch.cuda.current_stream().cuda_stream)
    assert torch.equal(out, gp.forward(m))
    assert torch.equal(gp.adjoint(d), want)


@pytest.mark.parametrize("how", ["adjoint", "stage", "solve"])
def test_after_a_failed_adjoint(case, how):
    """The large bound of the failed call does not reach the next one."""
    gp, _, d, want = case
    big = 1e6 * d
    call = {"adjoint": lambda: gp.adjoint(big),
            "stage": lambda: gp.apply_stage(4, gp.apply_stage(3, big)),
            "solve": lambda: gp.sparse_solve(big, 1.0, 3, gamma=1e-3, use_graph=False)}[how]
    _fail_adjoint(gp, call)
    assert torch.equal(gp.adjoint(d), want)
    assert torch.equal(gp.adjoint(d), want)


def test_capture_after_a_failed_adjoint(case):
    """An adjoint captured right after the failure clears the table when the
    graph runs; the direct call before that run clears it too."""
    gp, _, d, want = case
    _fail_adjoint(gp, lambda: gp.adjoint(1e6 * d))
    out = torch.empty_like(want)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        gp.adjoint(d, out)
    assert torch.equal(gp.adjoint(d), want)
    for _ in range(2):
        out.zero_()
        g.replay()
        assert torch.equal(out, want)
    assert torch.equal(gp.adjoint(d), want)
