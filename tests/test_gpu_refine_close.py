"""The end of a refinement (iod_refine): its cost is never above the start's by iod_eval's
evaluation, and belongs to the state returned: x0 with iod_eval's cost of it, or a refined
state with the FP64 sum of its squared residuals."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def fp64_cost(sc, ang, x):
    """The CHI2 cost of x by plain FP64 RK4 on the problem's grid."""
    from test_gpu_split_step import rk4
    s = rk4(sc.mu, np.stack([sc.chief, x], 1), sc.t, sc.dt, np.float64)
    d = s[:, :3, 1] - s[:, :3, 0]
    ba = ang[:, 0] - np.arctan2(d[:, 1], d[:, 0])
    ba -= 2 * np.pi * np.rint(ba / (2 * np.pi))
    bb = ang[:, 1] - np.arcsin(d[:, 2] / np.sqrt((d * d).sum(1)))
    return ((ba / sc.sigma[0]) ** 2).sum() + ((bb / sc.sigma[1]) ** 2).sum()


@pytest.mark.parametrize("scenario", [1, 2])
def test_at_the_rounding_floor(scenario):
    """Noise-free: swarm and refinement end at costs that are rounding alone."""
    from paper_2207_13175_gb300 import api
    from paper_2207_13175_gb300 import inputs as I
    sc = I.paper_table(scenario)
    ang, _ = api.simulate_obs(sc.mu, sc.chief, sc.deputy, sc.t, sc.noise)
    bounds = api.bounds_from_chief(sc.deputy, sc.r_max_km, sc.v_max_ms, I.L_KM, I.TU_S)
    with api.Problem(sc.mu, sc.chief, sc.t, ang, sc.sigma, bounds, api.options(dt=sc.dt)) as G:
        J = lambda x: float(G.eval(np.asarray(x)[None, :]).cpu()[0])  # noqa: E731
        G.run(sc.m, sc.iters, sc.w, sc.c1, sc.c2, sc.seed)
        x0 = G.result()["state"]
        for iters in (0, 50, 50):
            x, c, _ = G.refine(x0, iters)
            assert c <= J(x0) and J(x) <= J(x0)
            if np.array_equal(x, x0):
                assert c == J(x0)
            x0 = x


@pytest.mark.parametrize("m", [64, 700])
def test_refined_cost_is_the_fp64_sum(m):
    """With noise; swarms on FP64 steps (64) and on split steps."""
    import scenarios as S
    from paper_2207_13175_gb300 import inputs as I
    sc = I.paper_scale("halo", 0, noise=True)
    sc = sc.with_(t=sc.t[::8], noise=sc.noise[::8])
    pair = S.Pair(sc)
    pair.gpu.run(m, 3, sc.w, sc.c1, sc.c2, 1)
    r = pair.gpu.result()
    x, c, _ = pair.gpu.refine(r["state"], 40)
    assert c <= r["cost"]
    # the swarm's FP64 cost and this one round within 1e-8 of the minimum's cost (each angle to
    # 1e-10 of its sigma); the split evaluation of the state differs by 1.6e-8
    assert abs(c - fp64_cost(sc, np.stack([pair.ra, pair.dec], 1), x)) <= 1e-8 * c
    x2, c2, _ = pair.gpu.refine(x, 0)
    assert np.array_equal(x2, x)
    if m >= 256:
        assert c2 == float(pair.gpu.eval(x[None, :]).cpu()[0])
    else:
        assert c2 == c
    pair.close()
