"""Costs of far deputies at t = 0, where the line of sight's own angle is better known than the
split residuals' 1e-15 rad: as exact as an FP64 arctangent and arcsine."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PI = np.longdouble("3.14159265358979323846264338327950288")


# beyond 1/32 LU
@pytest.mark.parametrize("form,r", [("dopri5", 0.0315), ("dopri5", 0.3), ("dopri5", 2.0), ("er3bp", 0.0315),
                                    ("er3bp", 0.7), ("rk4", 0.126), ("rk4", 1.0), ("rk4-one-thread", 0.3)])
def test_far_residuals_are_fp64_exact(form, r):
    from paper_2207_13175_gb300 import api
    from paper_2207_13175_gb300 import inputs as I
    rng = np.random.default_rng(8)
    m, ra, dec, sig = 2000, 1.1, -0.4, 1e-3
    c = np.array(I.chief_orbits()["halo"]["state"], dtype=float)
    a, el = rng.uniform(-np.pi, np.pi, m), rng.uniform(-1.2, 1.2, m)
    X = np.tile(c, (m, 1))
    X[:, :3] += r * np.stack([np.cos(el) * np.cos(a), np.cos(el) * np.sin(a), np.sin(el)], 1)
    kw = {"dopri5": {"integrator": api.DOPRI5}, "er3bp": {"dynamics": api.ER3BP, "ecc": 0.0549},
          "rk4-one-thread": {"threads_per_particle": 1}}.get(form, {})
    b = api.bounds_from_chief(c, 500.0, 5.0, I.L_KM, I.TU_S)
    with api.Problem(I.MU, c, np.zeros(1), np.array([[ra, dec]]), (sig, sig), b, api.options(**kw)) as G:
        got = G.eval(X).cpu().numpy()
    d = X[:, :3].astype(np.longdouble) - c[:3].astype(np.longdouble)
    ba = np.longdouble(ra) - np.arctan2(d[:, 1], d[:, 0])
    ba = ba - 2 * PI * np.rint(ba / (2 * PI))
    bb = np.longdouble(dec) - np.arcsin(d[:, 2] / np.sqrt((d * d).sum(1)))
    J = (ba / sig) ** 2 + (bb / sig) ** 2
    # rounding: of the function's angle and the difference, below pi (an ulp, 2^-51, over
    # sqrt(12) each), of the line of sight (2^-52 over sqrt(12), through the arcsine's secant,
    # 2.8 at most) and three times of the sum
    ang = np.sqrt(2 * (2.0 ** -51 / np.sqrt(12)) ** 2 + (2.8 * 2.0 ** -52 / np.sqrt(12)) ** 2)
    tol = np.sqrt((4 * (ba * ba + bb * bb) * ang ** 2) / sig ** 4 + 3 * (J * 2.0 ** -53) ** 2)
    err = (got - J) / tol
    assert np.sqrt(np.mean(err.astype(float) ** 2)) <= 1.0, np.sqrt(np.mean(err.astype(float) ** 2))
