"""The (E, M) measurement inside the tail of a round and as a launch of its own (more walkers or
larger lattices): histograms equal the oracle's, with exchanges in between and afterwards."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# L: no full 16 sites, remainders of 16, several loads a lane; m: one walker, a warp each, two a
# warp, one more than the tail takes; 33^2 x 64 and 46^2 x 32 above 64 KB of lattices a window
@pytest.mark.parametrize("L,h,m", [(3, 1, 1), (5, 2, 16), (6, 3, 17), (7, 1, 32), (8, 2, 33), (23, 2, 3),
                                   (45, 2, 32), (46, 2, 32), (33, 1, 64)])
def test_measurement_routes_bit_exact(L, h, m):
    import oracle as O
    import paper_1402_2328_gb300.rewl as R
    g = R.REWL(0, L, h, 0.75, m, 1e-3, 0.8, seed=500 + L, interval=200)
    o = O.REWL(0, L, h, 0.75, m, 1e-3, 0.8, seed=500 + L, interval=200)
    g.init()
    assert o.init() == 0
    g.run(max_rounds=2)
    o.run(2)
    g.set_param("measure_em", 1)
    o.measure_em(True)
    g.step(3)
    o.run(3)
    assert np.array_equal(g.hist_em(), o.hist_em())
    assert g.hist_em().sum() == 3 * h * m
    a, b = g.state(), o.state()
    for f in ("spins", "k", "lng", "H"):
        assert np.array_equal(a[f], b[f]), f
    g.close()
