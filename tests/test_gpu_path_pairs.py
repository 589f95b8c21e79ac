"""The mixed path against the FP64 path (itself held to the oracle elsewhere) where the oracle
would take long, from a random state, with and without obstacles.

Fused passes: runs of time nodes that start and end inside a ragged tile (D = 2), blocks of
four and eight time nodes with a shorter last one (D = 3).  One iteration at the mixed
path's one-step bound; a second one, which starts from the residual that the pass left, at
the bound that the lock-step tests hold tens of iterations to.

Axes beyond 5,632 points, which neither the fast transforms nor the tensor-core passes take:
an iteration and the refined operator on the dense FP32 passes, at time axes of one to ten
groups of sixteen nodes."""
import numpy as np
import pytest

from gpu_util import ensure_built, pair, random_state, rel_err
from test_gpu_parity_mixed import centred, refined_tol, step_tol

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_built()


def two_paths(T, N, masked, rng):
    P = int(np.prod(N))
    r0, r1 = rng.random(P) + 0.05, rng.random(P) + 0.05
    mask = (rng.random(P) < 0.2) if masked else None
    out = [pair(len(N), T, N, r0, r1, mask=mask, prec=p, check_every=0) for p in ("mixed", "fp64")]
    q, al, beta = random_state(out[0][0], rng)
    q = q.astype(np.float32).astype(np.float64)   # q is stored in FP32 on the mixed path
    for _, _, s in out:
        s.dot_set_state(q, al, beta, 1.4)
    return out[0][2], out[1][2]


def step_and_compare(a, b, tol):
    for s in (a, b):
        s.dot_solve(tol=0.0, maxit=1)
    for x, y in zip(a.dot_get_state()[:3], b.dot_get_state()[:3]):
        assert rel_err(x, y) < tol


@pytest.mark.parametrize("T,N", [(20, [100, 60]), (31, [130, 97]), (40, [200, 131]), (64, [256, 250]),
                                 (40, [32, 30, 66]), (20, [50, 70, 70]), (18, [70, 63, 100])])
@pytest.mark.parametrize("masked", [False, True])
def test_fused_passes(T, N, masked):
    a, b = two_paths(T, N, masked, np.random.default_rng(70 + T))
    step_and_compare(a, b, step_tol(T, N))
    # the penalty and the residual stay: without checks the next iteration reuses f.r
    step_and_compare(a, b, 1e-4)
    a.close()
    b.close()


@pytest.mark.parametrize("T,N", [(2, [5640, 3]), (1, [3, 5641]), (100, [2, 5640]), (159, [5634, 2]), (2, [3, 5650, 4])])
def test_axes_beyond_the_fast_transforms(T, N):
    rng = np.random.default_rng(80 + T)
    a, b = two_paths(T, N, False, rng)
    step_and_compare(a, b, step_tol(T, N))
    rhs = rng.standard_normal((T + 1) * int(np.prod(N))).astype(np.float32).astype(np.float64)
    x, y = a.dot_poisson(rhs), b.dot_poisson(rhs)
    a.close()
    b.close()
    assert rel_err(centred(x), centred(y)) < refined_tol(T, N)
