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
from gpu_util import ensure_built, pair, rel_err

pytestmark = pytest.mark.gpu

GRIDS = [(1, [2, 3]), (2, [4, 5]), (3, [7, 8]), (31, [16, 9]), (32, [13, 17]), (63, [60, 121]), (5, [128, 34]),
         (4, [26, 256]), (3, [509, 4]), (2, [5, 512]), (219, [6, 4]), (220, [6, 4]), (1, [3, 2816]), (1, [2817, 2]),
         (4, [3, 11, 6]), (2, [10, 16, 25])]


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
