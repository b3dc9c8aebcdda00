"""A run of a small swarm captured into a CUDA graph before the chief's FP64 positions exist:
the graph gives the run's results, and its replays do not form the positions again."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_captured_small_run():
    import torch
    from paper_2207_13175_gb300 import api
    from paper_2207_13175_gb300 import inputs as I
    c = np.array(I.chief_orbits()["halo"]["state"], dtype=float)
    t = np.linspace(0.0, 7.0 * I.DAY_TU, 50)
    ang = np.stack([np.linspace(-3.0, 3.0, 50), np.linspace(-1.4, 1.4, 50)], 1)
    b = api.bounds_from_chief(c, 500.0, 5.0, I.L_KM, I.TU_S)
    make = lambda: api.Problem(I.MU, c, t, ang, (I.ARCSEC,) * 2, b, api.options(dt=5e-4))  # noqa: E731
    s = torch.cuda.Stream()

    def ms(f):
        s.synchronize()
        t0 = time.perf_counter()
        f()
        s.synchronize()
        return time.perf_counter() - t0

    with torch.cuda.stream(s), make() as G, make() as H:
        G.run(300, 1, seed=3)              # buffers; split steps: no FP64 chief yet
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            G.run(64, 0, seed=3)
        graph.replay()
        got = G.result()
        again = min(ms(graph.replay) for _ in range(3))
        H.run(64, 0, seed=3)
        ref = H.result()
        plain = min(ms(lambda: H.run(64, 0, seed=3)) for _ in range(3))
        x, y = G.refine(got["state"], 2), H.refine(ref["state"], 2)
    assert np.array_equal(got["state"], ref["state"]) and got["cost"] == ref["cost"]
    assert np.array_equal(x[0], y[0]) and x[1] == y[1]
    # the chief alone takes as long as the swarm: with it a replay would take twice the run
    assert again < 1.5 * plain, (again, plain)
