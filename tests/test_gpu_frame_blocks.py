"""Register-FFT blocks as plans of working size have them: several column pairs
to a block (2048-sample frames and shorter) and analysis blocks that take several
pairs in turn (4096 and 8192), with a part last block, cubes of odd column
counts and uneven odd folds.  Every cube against the FP64 oracle: operators (1e-4
relative L2) and two fused FISTA iterations (1e-3), the bounds of the parity
tests; every column of the stages (2e-6 in all, 1e-5 a column)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import fista, ops
from paper_2505_00387_gb300 import _lib as L
from paper_2505_00387_gb300 import synthetic as syn
from paper_2505_00387_gb300.plan import AahrtPlan

from gpu_util import dev, host, oracle_H, oracle_plan, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_00387_gb300 import build
    build.build()


# nt, samples a frame, curvatures, azimuths, folds; pairs a block, pairs in turn
# (model, data) on 152 SMs
CASES = [
    (200, 512, 25, 17, (427, 431, 425, 433, 429, 435), 8, 1, 1),
    (400, 1024, 25, 17, (431, 427, 433), 4, 1, 1),
    (800, 2048, 41, 5, (205, 207, 207), 2, 1, 1),
    (1600, 4096, 31, 31, (965,), 1, 2, 2),
    (1001, 4096, 31, 30, (931, 933, 929), 1, 4, 4),
    (3200, 8192, 31, 15, (365,), 1, 2, 2),
    (3200, 8192, 31, 30, (923,), 1, 4, 4),
]


def _column_pairs(cols):
    return sum((c + 1) // 2 for c in cols)


def _close_columns(a, b):
    assert rel(a, b) < 2e-6
    assert (np.linalg.norm(a - b, axis=0) / np.linalg.norm(b, axis=0)).max() < 1e-5


@pytest.mark.parametrize("nt,nfft,nq,nth,folds,pairs,turn_m,turn_d", CASES)
def test_blocks_of_working_plans(nt, nfft, nq, nth, folds, pairs, turn_m, turn_d):
    q0, dq = syn.q_axis(nq)
    gs = []
    for c, n in enumerate(folds):
        hx, hy = syn.disc_offsets(np.random.default_rng([97, c]), n, 1500.0)
        gs.append(syn.Gather(nt, 4.0 / nt, nt, nq, q0, dq, nth, hx, hy))
    gp = AahrtPlan.batched(gs)
    r2max = max(float(np.max(g.hx ** 2 + g.hy ** 2)) for g in gs)
    os_ = [oracle_plan(g, r2max=r2max) for g in gs]
    assert gp.info.nfft == nfft
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert L.aahrt_plan_test_frame_shape(gp.handle) == (pairs, turn_m, turn_d)
        # the last block is a part one on both sides
        assert _column_pairs([nq * nth] * len(gs)) % (pairs * turn_m)
        assert _column_pairs(folds) % (pairs * turn_d)
    rng = np.random.default_rng(98)
    m = [rng.standard_normal((nt, nq, nth)).astype(np.float32) for _ in gs]
    d = [rng.standard_normal((nt, n)).astype(np.float32) for n in folds]
    m_dev = dev(np.concatenate([x.ravel() for x in m]))
    d_dev = dev(np.concatenate([x.ravel() for x in d]))

    def cubes(flat, shapes):
        at = np.cumsum([0] + [int(np.prod(s)) for s in shapes])
        return [flat[at[i]:at[i + 1]].reshape(s) for i, s in enumerate(shapes)]

    fwd = cubes(host(gp.forward(m_dev)), [x.shape for x in d])
    adj = cubes(host(gp.adjoint(d_dev)), [x.shape for x in m])
    want = [ops.adjoint(p, x.astype(np.float64)) for p, x in zip(os_, d)]
    for c, p in enumerate(os_):
        assert rel(fwd[c], ops.forward(p, m[c].astype(np.float64))) < 1e-4
        assert rel(adj[c], want[c]) < 1e-4

    # two fused iterations: a step well below 1 / ||L||^2 and a threshold that
    # zeroes part of the model
    gamma = 0.2 / (nq * max(np.bincount(p.j0, minlength=nth).max() for p in os_))
    lam = 0.1 * max(float(np.abs(x).max()) for x in want)
    sol, _ = gp.sparse_solve(d_dev, lam, 2, gamma=gamma, want_info=False)
    for c, x in enumerate(cubes(host(sol), [x.shape for x in m])):
        ref = fista.solve(os_[c], d[c].astype(np.float64), lam, 2, gamma)
        assert 0.001 < np.count_nonzero(ref) / ref.size < 0.999
        assert rel(x, ref) < 1e-3

    # the analysis and synthesis blocks, column by column
    L.aahrt_plan_test_stage_frames(gp.handle, True)
    nb, C = os_[0].nbins, nq * nth
    X = cubes(host(gp.apply_stage(0, m_dev)), [(nb, C)] * len(gs))
    Y = cubes(host(gp.apply_stage(3, d_dev)), [(nb, n) for n in folds])
    Xc = torch.from_numpy(np.concatenate([x.astype(np.complex64).ravel() for x in X])).cuda()
    Yc = torch.from_numpy(np.concatenate([y.astype(np.complex64).ravel() for y in Y])).cuda()
    mt = cubes(host(gp.apply_stage(5, Xc)), [(nt, C)] * len(gs))
    dt = cubes(host(gp.apply_stage(2, Yc)), [(nt, n) for n in folds])
    for c, p in enumerate(os_):
        _close_columns(X[c], ops.rfft_bins(p, ops.stretch(p, m[c].reshape(nt, C).astype(np.float64))))
        _close_columns(Y[c], ops.rfft_bins(p, ops.unstretch_T(p, d[c].astype(np.float64))))
        _close_columns(mt[c], ops.stretch_T(p, oracle_H(p, X[c])))
        _close_columns(dt[c], ops.unstretch(p, oracle_H(p, Y[c])))
