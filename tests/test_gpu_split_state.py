"""States in FP32 words and back (iod_ff.cuh, to_state and from_state): an epoch at t = 0
returns the caller's states bit for bit, and a propagation of FP64 steps alone does not
depend on how many epochs it is handed over at."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def problem(chief, t, threads, **kw):
    from paper_2207_13175_gb300 import api
    from paper_2207_13175_gb300 import inputs as I
    b = api.bounds_from_chief(chief, 500.0, 5.0, I.L_KM, I.TU_S)
    K = len(t)
    return api.Problem(I.MU, chief, t, np.zeros((K, 2)) + 0.1, (I.ARCSEC,) * 2, b,
                       api.options(threads_per_particle=threads, **kw))


def halo():
    from paper_2207_13175_gb300 import inputs as I
    return np.array(I.chief_orbits()["halo"]["state"], dtype=float)


# quads of lanes up to 4,864 states, one thread each beyond and when asked for
@pytest.mark.parametrize("threads,m", [(0, 301), (1, 301), (0, 5000)])
def test_epoch_at_zero_returns_the_states(threads, m):
    from paper_2207_13175_gb300 import inputs as I
    rng = np.random.default_rng(5)
    X = rng.uniform(-1.0, 1.0, (m, 6))
    X[40:80, 0] *= 2.0 ** -rng.integers(1, 60, 40)              # x near the barycentre
    X[80:120] *= 2.0 ** -rng.integers(60, 1000, (40, 1))         # below FP32's range in part
    X[120:140] *= 2.0 ** rng.integers(3, 1000, (20, 1))          # far, and beyond FP32's range
    X[140:160, 0] = -I.MU + rng.uniform(0.05, 0.7, 20)           # near the Earth
    X[160:170, 0] = 1.0 - I.MU                                   # at the Moon's abscissa
    X[170:176] = np.where(np.eye(6, dtype=bool), np.inf, X[170:176])
    X[176:182] = 0.0
    with problem(halo(), np.array([0.0, 0.01]), threads) as G:
        out = G.propagate(X).cpu().numpy()
    assert np.array_equal(out[0], X.T)


@pytest.mark.parametrize("threads", [0, 1])
def test_fp64_steps_alone_are_the_same_over_any_epochs(threads):
    """Circular orbits 0.12-0.35 LU about the Earth at h = 2^-10 are too near for the split
    step; all epochs and steps are multiples of 2^-10, so the steps are the same ones."""
    from paper_2207_13175_gb300 import inputs as I
    rng = np.random.default_rng(6)
    m, h, n = 64, 2.0 ** -10, 160
    r, a = rng.uniform(0.12, 0.35, m), rng.uniform(-np.pi, np.pi, m)
    v = np.sqrt((1 - I.MU) / r) - r
    X = np.stack([-I.MU + r * np.cos(a), r * np.sin(a), 0.01 * r, -v * np.sin(a), v * np.cos(a), 0 * r], 1)
    last = []
    for K in (1, 5, 32, 160):
        t = h * np.arange(n // K, n + 1, n // K)
        with problem(halo(), t, threads, dt=h) as G:
            last.append(G.propagate(X).cpu().numpy()[-1])
    for q in last[1:]:
        assert np.array_equal(q, last[0]), np.max(np.abs(q - last[0]))


@pytest.mark.parametrize("threads", [0, 1])
def test_costs_of_states_that_words_do_not_hold(threads):
    """Costs at t = 0 of states that stay in FP64, and with a chief that does (its abscissa
    within 2^-18 of the barycentre), against the same formula here."""
    from paper_2207_13175_gb300 import api
    from paper_2207_13175_gb300 import inputs as I
    rng = np.random.default_rng(7)
    for x0 in (0.9, 3.0e-7):
        c = np.array([x0, 0.4, 0.1, 0.1, 0.2, 0.0])
        X = np.tile(c, (64, 1)) + rng.uniform(-1e-3, 1e-3, (64, 6))
        X[:16, 0] = rng.uniform(-1.0, 1.0, 16) * 2.0 ** -rng.integers(19, 70, 16)
        X[16:24, :3] *= 1e39
        with problem(c, np.zeros(1), threads) as G:
            J = G.eval(X).cpu().numpy()
        d = X[:, :3] - c[:3]
        ba, bb = 0.1 - np.arctan2(d[:, 1], d[:, 0]), 0.1 - np.arcsin(d[:, 2] / np.sqrt((d * d).sum(1)))
        ba -= 2 * np.pi * np.rint(ba / (2 * np.pi))
        ref = (ba * ba + bb * bb) / I.ARCSEC ** 2
        # residuals of 1e-2 rad and more, each side within a few 1e-14 rad
        assert np.allclose(J, ref, rtol=1e-10, atol=2 * 4e-14 ** 2 / I.ARCSEC ** 2), np.max(np.abs(J / ref - 1))
