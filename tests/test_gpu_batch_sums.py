"""The sum of squared beta increments of the fused D = 2 pass (k_fused2d.cu), which enters
eta_P^soc and so the penalty rule.

Its order is the grid's alone: a request in a batch reports the stopping measures of a
context, bit for bit.  And it takes every cell of every time node once, over runs of one to
eight nodes with a shorter last run, at each number of tile rows, with ragged tiles on both
axes, with and without obstacles.

Bound of the second test, on the sum: beta's update by inc is stored to 2^-48 of beta, from
tau inc rounded to FP32, so inc read off two states is right to 2^-23; the pass adds ten
squares per node of a run in FP32, each addition rounding a sum of positive terms by at
most u = 2^-24, and each square by u more (what follows is two-float and FP64).  The sum of the squares is then within
(10 run + 8) u of the one formed from the states."""
import numpy as np
import pytest

from gpu_util import ensure_built, pair, random_state
from paper_2505_05424_gb300 import workloads as W
from paper_2505_05424_gb300.solver import DotServer, DotSolver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_built()


# a small sigma keeps eta_P^soc above eta_P, so that the sum shows
@pytest.mark.parametrize("N,T", [(64, 32), (128, 32), (100, 20)])
@pytest.mark.parametrize("masked", [False, True])
def test_batch_reports_the_measures_of_a_context(N, T, masked):
    r0, r1, mask = W.mixture_pair(W.GridSpec(2, T, N), 4100, obstacles=masked)
    s = DotSolver(2, T, N, r0, r1, mask=mask, prec="mixed", sigma0=1e-3)
    s.dot_solve(tol=0.0, maxit=10)
    alone = s.dot_kkt()
    s.close()
    assert alone["eta_P_soc"] > alone["eta_P"]
    with DotServer(sigma0=1e-3) as srv:
        rid = srv.submit(2, T, N, r0, r1, mask=mask, tol=0.0, maxit=10, keep_fields=False)
        srv.wait(rid, 120.0)
        served = srv.result(rid)["kkt"]
    for k in ("eta_dot", "eta_P", "eta_D", "eta_C", "eta_P_soc", "eta_D_soc", "primal_obj", "dual_obj"):
        assert alone[k] == served[k], k


# rows and run: 4, 1 / 8, 1 / 13, 1 / 13, 2 (nine nodes) / 13, 4 (65) / 13, 8 (nine)
@pytest.mark.parametrize("T,N,masked", [(5, [33, 65], True), (20, [100, 60], False), (40, [200, 131], True),
                                        (8, [520, 515], False), (8, [520, 515], True), (64, [256, 250], False),
                                        (64, [256, 250], True), (8, [1000, 1023], False)])
def test_sum_takes_every_cell_once(T, N, masked):
    rng = np.random.default_rng(50 + T + N[1])
    P = int(np.prod(N))
    r0, r1 = rng.random(P) + 0.05, rng.random(P) + 0.05
    mask = (rng.random(P) < 0.2) if masked else None
    g, _, gpu = pair(2, T, N, r0, r1, mask=mask, prec="mixed", check_every=0)
    q, al, beta = random_state(g, rng)
    sigma, tau = 1.4, 1.9
    gpu.dot_set_state(q, al, beta, sigma)
    gpu.dot_solve(tol=0.0, maxit=1)
    b2 = gpu.dot_get_state()[2]
    soc = gpu.dot_kkt()["eta_P_soc"]
    gpu.close()
    vol = 1.0 / (T * P)
    want = ((b2 - beta) ** 2).sum() / (np.float32(tau).astype(float) * sigma) ** 2
    got = (soc * (1.0 + np.sqrt(vol * 2.0 * T * P))) ** 2 / vol
    assert abs(got - want) <= (10 * 8 + 8) * 2.0 ** -24 * want
