"""What reading fields back costs through the C ABI, against what it cannot do without: one
plain copy of each field into the caller's arrays and one multiplication of the densities
and momenta in place (rho = alpha_0 / h_0, m = alpha / h_0), timed here on the same arrays.
FP64 fields of a few MB, short enough for a fixed cost per call to show; a factor of two
leaves room for the padded rows of the momenta and for noise."""
import time

import numpy as np
import pytest

from gpu_util import ensure_built
from paper_2505_05424_gb300.solver import DotSolver, _dp

pytestmark = pytest.mark.gpu


def median_time(f, n=41):
    out = []
    for _ in range(n):
        t = time.perf_counter()
        f()
        out.append(time.perf_counter() - t)
    return float(np.median(out))


@pytest.mark.parametrize("T,N", [(32, 64), (16, 100)])
def test_fields_cost_their_copies(T, N):
    import torch
    ensure_built()
    rng = np.random.default_rng(8)
    s = DotSolver(2, T, N, rng.random((N, N)) + 0.1, rng.random((N, N)) + 0.1, prec="fp64")
    s.dot_solve(tol=0.0, maxit=4)
    rho, m, phi = np.ones(T * N * N), np.ones(2 * (T + 1) * N * (N - 1)), np.ones((T + 1) * N * N)
    dev = [torch.from_numpy(a).cuda() for a in (rho, m, phi)]

    def read():
        assert s.lib.dot_get(s.ctx, _dp(rho), _dp(m), _dp(phi), None, None) == 0

    def plain():
        for a, d in zip((rho, m, phi), dev):
            torch.from_numpy(a).copy_(d)
        np.multiply(rho, 1.0, out=rho)
        np.multiply(m, 1.0, out=m)

    read()
    plain()
    whole, needed = median_time(read), median_time(plain)
    s.close()
    print(f"dot_get {1e6 * whole:.0f} us, copies and scaling {1e6 * needed:.0f}")
    assert whole <= 2.0 * needed
