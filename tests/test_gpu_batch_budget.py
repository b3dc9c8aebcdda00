"""The batch's memory accounting against what it asks of its allocator: the bytes in use and
their high water are the bytes requested for the resident problems, table by table, and a
budget one byte below a request's allocation refuses it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def request(K, m, iters=2):
    from paper_2207_13175_gb300 import api
    from paper_2207_13175_gb300 import inputs as I
    c = np.array(I.chief_orbits()["halo"]["state"], dtype=float)
    t = np.linspace(0.0, 0.2, K)
    ang = np.stack([np.linspace(-3.0, 3.0, K), np.linspace(-1.4, 1.4, K)], 1)
    b = api.bounds_from_chief(c, 250.0, 2.0, I.L_KM, I.TU_S)
    return (I.MU, c, t, ang, (I.ARCSEC,) * 2, b, m, iters, 0.7, 1.5, 1.5, 3)


# many epochs beside few particles and the reverse; with the FP64 chief (small swarms,
# refinements) and without
@pytest.mark.parametrize("K,m", [(400, 8), (400, 300), (3, 2000)])
@pytest.mark.parametrize("kw", [dict(), dict(precision=1), dict(refine_iters=2)])
def test_bytes_in_use_are_the_bytes_allocated(K, m, kw):
    from paper_2207_13175_gb300 import api
    from test_gpu_failures import FlakyAllocator
    with FlakyAllocator() as A:
        B = api.Batch(api.options(dt=1e-3, **kw), budget_bytes=1 << 30, max_resident=4, torch_allocator=False)
        before = dict(A.live)
        t0 = B.submit(*request(K, m))
        B.step(0)
        st = B.stats()
        sizes = {p: n for p, n in A.live.items() if p not in before}
        assert st["resident"] == 1
        assert st["bytes_in_use"] == max(sizes.values()) == st["bytes_high_water"], (st, sizes)
        one = st["bytes_in_use"]
        B.cancel(t0)
        B.close()
        for budget in (one, one - 1):
            B = api.Batch(api.options(dt=1e-3, **kw), budget_bytes=budget, max_resident=4, torch_allocator=False)
            if budget == one:
                B.submit(*request(K, m))
            else:
                with pytest.raises(api.IodError) as e:
                    B.submit(*request(K, m))
                assert e.value.code == -2
            B.close()
