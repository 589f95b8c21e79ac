"""Axes with a large prime factor p: their transforms cost p multiply-adds per output, so
the fast Poisson solve (k_fft.cu) has to be no worse there than the dense transforms that
the library also has.  Device times of one process.

FP32: the solve of an iteration on 508 = 4 x 127 points against a solve of dot_poisson, which
runs the dense passes on the tensor cores; 1.5 for their better unit.  FP64: an iteration's
solve on 2801 (prime, the fast form) against 2820 points (the dense form)."""
import numpy as np
import pytest

from gpu_util import ensure_built
from paper_2505_05424_gb300.solver import DotSolver
from test_gpu_fast_poisson import one_iteration

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_built()


# four outputs per thread: the last group with two (67, 131), one (73) and three (509) of
# them, both kinds of axis, eight and four pairs per block; and two per thread (37, 61, 101)
@pytest.mark.parametrize("T,N", [(20, [268, 292]), (8, [509, 524]), (3, [37, 61, 101])])
def test_fp32_iteration(T, N):
    """At the mixed path's one-step bound."""
    one_iteration(T, N)


def transforms_ms(s, run, solves):
    """Time of the transform and scale kernels per solve, best of three."""
    run()
    best = np.inf
    for _ in range(3):
        s.dot_profile(True)
        run()
        k = s.dot_profile_read()
        best = min(best, sum(k[n][0] for n in ("dct_axis", "dct_scale", "dct_tcgen05")) / solves)
        s.dot_profile(False)
    return best


def solver(T, N, prec):
    rng = np.random.default_rng(12)
    return DotSolver(2, T, N, rng.random(N) + 0.1, rng.random(N) + 0.1, prec=prec, check_every=0)


def iteration_ms(s):
    return transforms_ms(s, lambda: s.dot_solve(tol=0.0, maxit=10), 10)


def test_fp32_against_the_dense_passes():
    s = solver(32, [508, 508], "mixed")
    b = np.random.default_rng(13).standard_normal(33 * 508 * 508)
    dense = transforms_ms(s, lambda: s.dot_poisson(b), 2)    # a solve and its refinement
    fast = iteration_ms(s)
    s.close()
    print(f"508^2 x 32: fast {1e3 * fast:.0f} us, dense {1e3 * dense:.0f} us")
    assert fast <= 1.5 * dense


def test_fp64_against_the_dense_passes():
    ms = []
    for n in (2801, 2820):
        s = solver(2, [n, 4], "fp64")
        ms.append(iteration_ms(s))
        s.close()
    print(f"2801: fast {1e3 * ms[0]:.0f} us, 2820: dense {1e3 * ms[1]:.0f} us")
    assert ms[0] <= ms[1]
