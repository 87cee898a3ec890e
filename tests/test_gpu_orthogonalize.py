"""The orthogonalisation kernels (Algorithm 1's LQ sweep and QR steps, ranks up to 32 in one kernel
family) against the oracle at the edges of their tiles: ranks at and around multiples of four, square
unfoldings, one row more than a pass of 512 threads takes, neighbours that do not fit beside the
unfolding, ranks above 32 (the kernels for larger ranks) among smaller ones, wide and rank-deficient
unfoldings inside a sweep (Householder). Tolerances are the suite's: 1e-4 for cores (the gauge
amplifies rounding), 1e-5 for the tensor."""
import numpy as np
import pytest

import tt_oracle as O
from paper_2309_08093_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2309_08093_gb300 import build as _build  # noqa: E402

_build.build()
from paper_2309_08093_gb300 import lib  # noqa: E402


def rel(a, b):
    return np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel())


@pytest.mark.parametrize("dims,ranks", [
    ((50, 50), (1, 4, 1)), ((50, 40), (1, 5, 1)), ((40, 30, 20), (1, 8, 9, 1)), ((40, 30, 20), (1, 13, 17, 1)),
    ((60, 30, 40), (1, 21, 24, 1)), ((60, 20, 50), (1, 25, 20, 1)), ((64, 12, 70), (1, 32, 16, 1)),
    ((12, 6, 12), (1, 12, 12, 1)),            # square end unfoldings
    ((513, 10, 5), (1, 4, 5, 1)), ((1025, 6), (1, 6, 1)),  # one row past one and two per thread
    ((3300, 10, 9), (1, 12, 8, 1)),           # no room for the neighbour beside the unfolding
    ((40, 40, 20), (1, 33, 12, 1)),           # a rank above 32 beside a smaller one
    ((7, 2, 3, 2, 7), (1, 6, 12, 6, 6, 1)),   # a wide unfolding on the way left to right
])
def test_sweep_and_steps(dims, ranks):
    cores = synth.random_tt(dims, ranks, 77)
    c32 = [np.asarray(g, np.float32).astype(np.float64) for g in cores]
    ctx = lib.Context(dims, ranks, 64, 1e-3, 5)
    dc = lib.device_cores(cores)
    ctx.tt_orthogonalize(dc, -1)
    got, ref = lib.host_cores(dc, ranks, dims), O.orthogonalize_right_to_left(c32)
    for g, r in zip(got, ref):
        assert rel(g, r) <= 1e-4
    for k in range(len(dims) - 1):
        ctx.tt_orthogonalize(dc, +1, k)
        O.left_orthogonalize_step(ref, k)
        got = lib.host_cores(dc, ranks, dims)
        m, q = ranks[k] * dims[k], ranks[k + 1]
        if m >= q:
            assert rel(got[k], ref[k]) <= 1e-4 and rel(got[k + 1], ref[k + 1]) <= 1e-4
        GL = got[k].reshape(m, q, order="F")[:, :min(m, q)]
        assert np.allclose(GL.T @ GL, np.eye(min(m, q)), atol=1e-5)
        ref = [g.copy() for g in got]  # (a wide unfolding's Q is not unique)
    assert rel(O.tt_full(got), O.tt_full(c32)) <= 1e-5
    ctx.close()


def test_rank_deficient_core_inside_the_sweep():
    """A repeated slice makes the middle unfolding rank deficient: the sweep's second step falls back to
    Householder on the core that the first step left in shared memory."""
    dims, ranks = (9, 7, 6), (1, 5, 6, 1)
    cores = synth.random_tt(dims, ranks, 41)
    cores[1][4] = cores[1][1]
    c32 = [np.asarray(g, np.float32).astype(np.float64) for g in cores]
    ctx = lib.Context(dims, ranks, 64, 1e-3, 5)
    dc = lib.device_cores(cores)
    ctx.tt_orthogonalize(dc, -1)
    got = lib.host_cores(dc, ranks, dims)
    assert rel(O.tt_full(got), O.tt_full(c32)) <= 1e-5
    for g in got[1:]:
        GR = g.reshape(g.shape[0], -1, order="F")
        assert np.allclose(GR @ GR.T, np.eye(GR.shape[0]), atol=1e-5)
    ctx.close()
