"""The boundary scale (y_0 + |ybar|) / (2 |ybar|) of the cone projection (ffloat.cuh), which
multiplies every component, is as good as its own roundings.

From q = alpha = 0 and a large sigma the projection's input is d - beta/sigma alone (the
potential is of the order of 1 / sigma).  The scale's error of a cone is the common part
of its components' errors, read off beta's update against the oracle's.  In units of
u = 2^-24: the numerator, |ybar| and the quotient are rounded once each, 0.42 rms for a
mantissa log-uniform in [1, 2); the roundings of thirteen components of z and of the faces'
q average out to 0.12 and 0.15.  Together 0.76; a fourth error of a rounding's size would
make it 0.87.  The bound lies halfway."""
import numpy as np
import pytest

import oracle as O
from gpu_util import ensure_built, pair

pytestmark = pytest.mark.gpu


def test_boundary_scale_is_rounded_once():
    ensure_built()
    T, N, K = 6, [16, 15, 14], 14
    P = int(np.prod(N))
    rng = np.random.default_rng(5)
    g, prob, gpu = pair(3, T, N, np.ones(P), np.ones(P), prec="mixed", check_every=0)
    sigma, tau = 2.0 ** 27, 1.9
    B = rng.standard_normal((K, T * P))
    q, al, beta = np.zeros(g.n_q), np.zeros(g.n_q), (B * sigma).ravel()
    st = O.State(g, np.zeros(g.n_nodes), np.zeros(K * g.n_cones), q.copy(), al.copy(), beta.copy(), sigma)
    O.iterate(prob, st, tau=tau)
    gpu.dot_set_state(q, al, beta, sigma)
    gpu.dot_solve(tol=0.0, maxit=1)
    got = gpu.dot_get_state()[2]
    gpu.close()
    err = ((got - st.beta) / (float(np.float32(tau)) * sigma)).reshape(K, -1)
    y = -B
    y[0] += 1.0
    y[K - 1] += 1.0
    n2 = (y[1:] ** 2).sum(0)
    edge = np.abs(y[0]) < np.sqrt(n2)
    scale = 0.5 * (y[0] + np.sqrt(n2)) / np.sqrt(n2)
    e = ((err[1:] * y[1:]).sum(0) / n2 / scale)[edge] * 2.0 ** 24
    print(f"{edge.sum()} cones, rms {np.sqrt((e ** 2).mean()):.3f} u")
    assert np.sqrt((e ** 2).mean()) <= 0.815
