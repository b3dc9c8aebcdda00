"""Where the split FP32 RK4 step gives way to FP64 steps (iod_ff.cuh, make_step): near the
Earth, at the Moon and for other mass parameters, circular orbits about either primary against
the same RK4 in extended precision are no less exact than a plain FP64 implementation."""
import math

import numpy as np
import pytest

from test_gpu_split_step import rk4

pytestmark = pytest.mark.gpu

EM = 0.01215058560962404


def circular(mu, moon, r, m, seed=0):
    """States [m][6] on circular orbits of radius r about a primary, every inclination."""
    rng = np.random.default_rng(seed)
    a = rng.normal(size=(m, 3))
    a /= np.linalg.norm(a, axis=1)[:, None]
    b = rng.normal(size=(m, 3))
    b -= (a * b).sum(1)[:, None] * a
    b /= np.linalg.norm(b, axis=1)[:, None]
    rr = r * (1 + 0.02 * rng.uniform(-1, 1, m))[:, None]
    v = np.sqrt((mu if moon else 1 - mu) / rr) * b
    p = rr * a
    v[:, 0] += p[:, 1]                       # rotating frame
    v[:, 1] -= p[:, 0]
    p[:, 0] += (1 - mu) if moon else -mu
    return np.concatenate([p, v], 1)


@pytest.mark.parametrize("mu,moon,r,h,T", [
    (EM, 0, 0.26, 2.5e-4, 0.46), (EM, 0, 0.17, 1e-4, 0.3), (EM, 0, 0.12, 5e-5, 0.15), (EM, 0, 0.08, 1e-5, 0.03),
    (EM, 0, 0.36, 5e-4, 0.46), (3e-6, 0, 0.36, 5e-4, 0.46), (3e-6, 0, 0.8, 5e-4, 1.6), (0.3, 0, 0.36, 5e-4, 0.46),
    (EM, 0, 0.65, 5e-4, 0.46), (EM, 0, 0.9, 1e-3, 0.46), (EM, 1, 0.05, 2e-3, 0.05), (EM, 1, 0.024, 5e-4, 0.05),
    (EM, 1, 0.1, 2e-3, 0.46), (3e-6, 1, 0.003, 1e-3, 0.46), (0.4, 1, 0.3, 2e-3, 0.46)])
def test_circular_orbits_are_as_exact_as_fp64(mu, moon, r, h, T):
    from paper_2207_13175_gb300 import api
    from paper_2207_13175_gb300 import inputs as I
    n, K = round(T / h), 10
    h = 2.0 ** -40 * round(h * 2.0 ** 40)    # the same steps on both sides
    t = h * np.array([math.ceil(n * (k + 1) / K) for k in range(K)])
    X = circular(mu, moon, r, 48)
    ref = rk4(mu, X.T, t, h, np.longdouble)
    e64 = (rk4(mu, X.T, t, h, np.float64) - ref).astype(float)
    c = circular(mu, moon, r, 1, seed=9)[0]
    b = api.bounds_from_chief(c, 500.0, 5.0, I.L_KM, I.TU_S)
    with api.Problem(mu, c, t, np.zeros((K, 2)) + 0.1, (I.ARCSEC,) * 2, b, api.options(dt=h)) as G:
        got = G.propagate(X).cpu().numpy()
    eg = (got - ref).astype(float)
    # as in test_gpu_split_step: a quarter between two FP64 implementations, outputs to 2^-54
    rms = lambda e: math.sqrt(float(np.mean(e[:, :3] ** 2)))  # noqa: E731
    assert rms(eg) <= 1.25 * rms(e64) + 2.0 ** -54, (rms(eg), rms(e64))
