"""The fast Poisson solve (k_fft.cu) through the FP64 operator entry point, against the
oracle's dense transforms: axis lengths of every radix (2, 3, 4, 5, 8, other primes and
their products), the shortest and longest that fit the kernel and the first that does
not, odd and even row counts; time axes of one to several nodes per lane and around
the longest that fits.

Bound: each of the two solves rounds at u = 1.1e-16 with an amplification of at most
the Neumann Laplacian's condition number (2 n / pi)^2 on the longest axis; ten such
roundings and the 1e-13 of short axes' sums."""
import numpy as np
import pytest

import oracle as O
from gpu_util import ensure_built, pair, random_state, rel_err
from test_gpu_parity_mixed import step_tol

pytestmark = pytest.mark.gpu

GRIDS = [(1, [2, 3]), (2, [4, 5]), (3, [7, 8]), (31, [16, 9]), (32, [13, 17]), (63, [60, 121]), (5, [128, 34]),
         (4, [26, 256]), (3, [509, 4]), (2, [5, 512]), (219, [6, 4]), (220, [6, 4]), (1, [3, 2816]), (1, [2817, 2]),
         (4, [3, 11, 6]), (2, [10, 16, 25]),
         # axes of 64 .. 1024 with just enough (and a few more) sequences for the compile-time form
         (75, [64, 128]), (37, [256, 64]), (18, [512, 128]), (1, [1024, 608]), (1, [609, 1024]), (3, [608, 512]),
         (3, [609, 256])]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_built()


@pytest.mark.parametrize("T,N", GRIDS)
def test_fp64_poisson(T, N):
    rng = np.random.default_rng(40 + T + sum(N))
    g = O.Grid(len(N), T, N)
    b = rng.standard_normal(g.n_nodes) + 0.5
    r0 = rng.random(int(np.prod(N))) + 0.1
    gpu = pair(len(N), T, N, r0, r0, prec="fp64")[2]
    phi = gpu.dot_poisson(b)
    gpu.close()
    n = max([T + 1] + list(N))
    assert rel_err(phi, O.poisson(g, b)) < 1e-13 + 1.1e-15 * (2 * n / np.pi) ** 2


@pytest.mark.parametrize("T,N", [(75, [64, 128]), (3, [512, 608]), (1, [4, 9, 600]), (2, [64, 76, 64])])
def test_fp32_iteration(T, N):
    """The FP32 form inside one iteration of the mixed path, at the mixed path's one-step
    bound."""
    one_iteration(T, N)


# the kernel of small grids (x transforms and time solve in one block): its smallest, the
# largest by (T + 1) N_x and the next, odd N_y (half a pair), prime and even T + 1, the
# longest time axis, and short ones whose x axis just fits and does not fit its memory
@pytest.mark.parametrize("T,N", [(1, [2, 2]), (1, [3, 5]), (16, [512, 5]), (16, [513, 4]), (37, [229, 7]),
                                 (159, [54, 31]), (40, [31, 2]), (1, [4020, 3]), (1, [4032, 2])])
def test_fp32_iteration_small(T, N):
    """As above."""
    one_iteration(T, N)


def one_iteration(T, N):
    rng = np.random.default_rng(70 + T + sum(N))
    D, P = len(N), int(np.prod(N))
    r0, r1 = rng.random(P) + 0.05, rng.random(P) + 0.05
    g, prob, gpu = pair(D, T, N, r0, r1, prec="mixed", check_every=0)
    q, al, beta = random_state(g, rng)
    q = q.astype(np.float32).astype(np.float64)   # q is stored in FP32 on the GPU
    st = O.State(g, np.zeros(g.n_nodes), np.zeros(g.K * g.n_cones), q.copy(), al.copy(), beta.copy(), 1.3)
    O.iterate(prob, st, tau=1.9)
    gpu.dot_set_state(q, al, beta, 1.3)
    gpu.dot_solve(tol=0.0, maxit=1)
    q2, al2, b2, _, _ = gpu.dot_get_state()
    phi = gpu.dot_get()[2].ravel()
    gpu.close()
    tol = step_tol(T, N)
    assert rel_err(phi - phi.mean(), st.phi) < tol
    assert rel_err(q2, st.q) < tol
    assert rel_err(al2, st.alpha) < tol
    assert rel_err(b2, st.beta) < tol
