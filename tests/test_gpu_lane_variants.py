"""Quads of lanes (split steps) and lane pairs (FP64 steps: swarms below 256 particles, steps
above 2.1e-3 TU) against one thread per particle with every variant of the swarm, at sizes
where they run: equal bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

L_KM = 384400.0
VARIANTS = {
    "tolerance": dict(tol_tau=1e-3),
    "constriction": dict(constriction=1, init_grid=1, velocity_init=1, per_dim_random=1),
    "cone": dict(init_cone=1, cone_rho_min=5.0 / L_KM, cone_rho_max=150.0 / L_KM),
    "quartic": dict(cost_form=1, vmax_frac=0.5),
    "range": dict(use_range=1, sigma_range=0.01 / L_KM),
}


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("variant", list(VARIANTS))
# quads; pairs for a small swarm; pairs for long steps
@pytest.mark.parametrize("m,dt,lanes", [(601, 1e-3, 0), (255, 1e-3, 2), (601, 4e-3, 2)])
def test_lanes_equal_one_thread(m, dt, lanes, variant, order):
    import scenarios as S
    from paper_2207_13175_gb300 import api
    from paper_2207_13175_gb300 import inputs as I
    sc = I.tiny(0)
    pair = S.Pair(sc)
    kw = VARIANTS[variant]
    coef = (1.0, 2.05, 2.05) if kw.get("constriction") else (sc.w, sc.c1, sc.c2)
    out = []
    for threads in (1, lanes):
        opts = api.options(dt=dt, gbest_order=order, threads_per_particle=threads, **kw)
        with api.Problem(sc.mu, sc.chief, sc.t, np.stack([pair.ra, pair.dec], 1), sc.sigma, pair.bounds, opts,
                         ranges=pair.rng if kw.get("use_range") else None) as G:
            G.run(m, 12, *coef, sc.seed)
            out.append((G.result(), G.swarm_get()))
    (a, sa), (q, sq) = out
    assert a["iters_done"] == q["iters_done"] and a["rk_steps"] == q["rk_steps"]
    assert np.array_equal(a["state"], q["state"]) and np.array_equal(a["gcost_trace"], q["gcost_trace"])
    assert np.array_equal(a["gidx_trace"], q["gidx_trace"])
    for k in ("x", "v", "p", "pJ", "J"):
        assert np.array_equal(sa[k], sq[k]), k
    pair.close()
