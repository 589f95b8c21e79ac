"""Reading a solve back (dot_get, dot_get_state) on the calling thread and, above 4 MB,
by several: padded face rows wider than a chunk, narrow ones with a remainder, both
precisions, two and three dimensions.  The state written is the state read: exactly in
FP64; in the mixed path q to FP32, the multipliers to the two-float's 2^-48 (and one
rounding each way through sigma)."""
import numpy as np
import pytest

import oracle as O
from gpu_util import ensure_built, pair, random_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_built()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("D,T,N", [(2, 3, [5, 7]), (2, 9, [260, 300]), (2, 40, [131, 70]), (3, 7, [30, 41, 37])])
def test_state_and_fields_round_trip(prec, D, T, N):
    rng = np.random.default_rng(11 + T)
    P = int(np.prod(N))
    r0 = rng.random(P) + 0.1
    g, _, gpu = pair(D, T, N, r0, r0, prec=prec)
    q, al, beta = random_state(g, rng)
    sigma = 0.37
    gpu.dot_set_state(q, al, beta, sigma)
    q2, al2, b2, s2, _ = gpu.dot_get_state()
    rho, m, phi, _, _ = gpu.dot_get()
    gpu.close()
    assert s2 == sigma
    if prec == "fp64":
        assert np.array_equal(q2, q) and np.array_equal(al2, al) and np.array_equal(b2, beta)
    else:
        assert np.array_equal(q2, q.astype(np.float32).astype(np.float64))
        assert np.abs(al2 - al).max() <= 2.0 ** -46 * np.abs(al).max()
        assert np.abs(b2 - beta).max() <= 2.0 ** -46 * np.abs(beta).max()
    n0 = g.n_cones
    assert np.array_equal(rho.ravel(), al2[:n0] * T)
    assert np.array_equal(np.concatenate([v.ravel() for v in m]), al2[n0:] * T)
    assert not phi.any()
