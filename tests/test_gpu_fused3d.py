"""The D = 3 passes (k_fused3d.cu): 4 x 4 x 32 tiles with ragged edges on every axis, one
and several time nodes per block, with and without obstacles.

Two iterations from a random state against the oracle: the second one starts from the
residual that the pass left.  The bound is the one that the mixed path's lock-step
tests hold tens of iterations to (1e-4 of each field's maximum)."""
import numpy as np
import pytest

import oracle as O
from gpu_util import ensure_built, pair, random_state, rel_err

pytestmark = pytest.mark.gpu

GRIDS = [(1, [2, 2, 2]), (3, [4, 4, 32]), (5, [5, 9, 33]), (20, [9, 8, 64]), (33, [6, 3, 31]), (2, [13, 5, 70]),
         (40, [32, 30, 66])]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_built()


@pytest.mark.parametrize("T,N", GRIDS)
@pytest.mark.parametrize("masked", [False, True])
def test_two_iterations_from_random_state(T, N, masked):
    rng = np.random.default_rng(300 + T + 7 * masked)
    P = int(np.prod(N))
    r0, r1 = rng.random(P) + 0.05, rng.random(P) + 0.05
    mask = (rng.random(P) < 0.2) if masked else None
    g, prob, gpu = pair(3, T, N, r0, r1, mask=mask, prec="mixed", check_every=0)
    q, al, beta = random_state(g, rng)
    q = q.astype(np.float32).astype(np.float64)   # q is stored in FP32 on the GPU
    sigma = 1.4
    st = O.State(g, np.zeros(g.n_nodes), np.zeros(g.K * g.n_cones), q.copy(), al.copy(), beta.copy(), sigma)
    for _ in range(2):
        O.iterate(prob, st, tau=1.9)
    gpu.dot_set_state(q, al, beta, sigma)
    gpu.dot_solve(tol=0.0, maxit=2)
    q2, al2, b2, _, it = gpu.dot_get_state()
    ko, kg = O.kkt(prob, st), gpu.dot_kkt()
    gpu.close()
    assert it == 2
    assert rel_err(q2, st.q) < 1e-4
    assert rel_err(al2, st.alpha) < 1e-4
    assert rel_err(b2, st.beta) < 1e-4
    for name in ("eta_P", "eta_D", "eta_C", "eta_P_soc", "eta_D_soc"):
        assert abs(kg[name] - ko[name]) <= 1e-3 * abs(ko[name]) + 1e-6, name
