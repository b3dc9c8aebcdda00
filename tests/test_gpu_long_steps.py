"""Problems whose steps are too long for the split step (above 2.1e-3 TU) keep to FP64 steps:
one thread, lane pairs, the balanced schedule, evaluation, the allocation-free scoring and
batches give the same costs, and states are those of plain FP64 RK4."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def setup(T=1.0, K=21, t=None):
    from paper_2207_13175_gb300 import api
    from paper_2207_13175_gb300 import inputs as I
    c = np.array(I.chief_orbits()["halo"]["state"], dtype=float)
    t = np.linspace(0.0, T, K) if t is None else t
    ang = np.stack([np.linspace(-3.0, 3.0, len(t)), np.linspace(-1.4, 1.4, len(t))], 1)
    return c, t, ang, api.bounds_from_chief(c, 500.0, 5.0, I.L_KM, I.TU_S)


def problem(s, **kw):
    from paper_2207_13175_gb300 import api
    from paper_2207_13175_gb300 import inputs as I
    c, t, ang, b = s
    return api.Problem(I.MU, c, t, ang, (I.ARCSEC,) * 2, b, api.options(**kw))


# seven eighths of the steps long (the rest in short intervals), and just fewer
def mixed_times(n_long, n_short):
    return np.cumsum([0.0] + [0.012] * n_long + [0.002] * n_short)       # 3 long steps or one short one


@pytest.mark.parametrize("dt,t,m", [(4e-3, None, 300), (2.5e-3, None, 4097), (4e-3, mixed_times(7, 3), 300),
                                    (4e-3, mixed_times(6, 3), 300), (8e-3, None, 20000)])
@pytest.mark.parametrize("order", [0, 1])
def test_every_form_gives_the_same_costs(dt, t, m, order):
    from paper_2207_13175_gb300 import api
    s = setup(t=t)
    out = []
    for kw in (dict(), dict(threads_per_particle=1, schedule=1),
               dict(threads_per_particle=2), dict(threads_per_particle=1, schedule=2)):
        with problem(s, dt=dt, gbest_order=order, **kw) as G:
            G.run(m, 3, 0.7, 1.5, 1.5, 5)
            sw = G.swarm_get()
            G.run(m, 0, 0.7, 1.5, 1.5, 5)
            x = G.swarm_get()
            assert np.array_equal(G.eval(x["x"].T).cpu().numpy(), x["J"])
            out.append((sw, G.chief_positions()))
    for sw, rc in out[1:]:
        for k in ("x", "p", "pJ", "J"):
            assert np.array_equal(sw[k], out[0][0][k]), k
        assert np.array_equal(rc, out[0][1])


def test_states_are_plain_fp64_rk4():
    from paper_2207_13175_gb300 import inputs as I
    from test_gpu_split_step import rk4
    s = setup(T=0.8, K=5)
    X = I.particles_in_box(s[3][:6], s[3][6:], 40, seed=2)
    X[0] = s[0]
    with problem(s, dt=4e-3) as G:
        got, rc = G.propagate(X).cpu().numpy(), G.chief_positions()
    assert np.array_equal(got[0], X.T) and np.array_equal(got[:, :3, 0], rc)
    assert np.max(np.abs(got - rk4(I.MU, X.T, s[1], 4e-3, np.float64))) <= 1e-12


def test_batches_and_scoring():
    import torch
    from paper_2207_13175_gb300 import _native as N
    from paper_2207_13175_gb300 import api
    from paper_2207_13175_gb300 import inputs as I
    s = setup()
    c, t, ang, b = s
    for precision in (0, 1):
        opts = dict(dt=4e-3, precision=precision, fp64_last_iters=2)
        B = api.Batch(api.options(**opts), budget_bytes=1 << 28, max_resident=4)
        tk = B.submit(I.MU, c, t, ang, (I.ARCSEC,) * 2, b, 500, 4, 0.7, 1.5, 1.5, 9)
        B.run()
        r = B.poll(tk)
        B.close()
        with problem(s, **opts) as G:
            G.run(500, 4, 0.7, 1.5, 1.5, 9)
            a = G.result()
        assert np.array_equal(r["state"], a["state"]) and r["cost"] == a["cost"]
    X = I.particles_in_box(b[:6], b[6:], 777, seed=4)
    with problem(s, dt=4e-3) as G:
        J, rc = G.eval(X).cpu().numpy(), G.chief_positions()
    obs = torch.from_numpy(np.concatenate([t[None], ang.T, rc.T]).copy()).to("cuda")
    d_x = torch.from_numpy(X.T.copy()).to("cuda")
    d_J, best = torch.empty(777, dtype=torch.float64, device="cuda"), torch.empty(8, dtype=torch.float64, device="cuda")
    p = lambda a: ctypes.c_void_p(a.data_ptr())  # noqa: E731
    assert N.lib().iod_score_noalloc(I.MU, len(t), p(obs), I.ARCSEC, I.ARCSEC, 4e-3, p(d_x), 777, p(d_J), p(best),
                                     None) == 0
    torch.cuda.synchronize()
    assert np.array_equal(d_J.cpu().numpy(), J) and float(best[0]) == J.min()
