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


# one window, fewer and more pairs than the CTA that picks the join points has warps, fewer and more points
# than it has partial sums for (1024 x 256).  The norm: a sum of n <= 4e5 positive terms of 2^-53 relative
# rounding each, far below 1e-11 of ln g.
@pytest.mark.parametrize("B,N1,h", [(12, 2, 1), (36, 9, 3), (300, 5, 40), (64, 700, 2), (401, 1001, 9)])
def test_join_em_sizes(B, N1, h):
    import torch
    import oracle as O
    import paper_1402_2328_gb300.rewl as R
    lo, hi = O.windows(B, h, 0.75)
    W = int((hi - lo).max()) + 1
    rng = np.random.default_rng(B)
    kk, jj = np.meshgrid(np.arange(B + 1) / B, np.arange(N1) / N1, indexing="ij")
    base = 40 * np.sin(2.1 * kk + 0.3) * np.cos(1.3 * jj - 0.2) + 9 * kk * jj
    S = np.full((h, W, N1), -np.inf)
    for w in range(h):
        S[w, : hi[w] - lo[w] + 1] = base[lo[w]: hi[w] + 1] + rng.normal(0, 10) + rng.normal(
            0, 1e-3, (hi[w] - lo[w] + 1, N1))
    S[rng.random(S.shape) < 0.05] = -np.inf
    ref, jref = O.join_em(lo, hi, S, B, N1 - 1)
    out = torch.zeros((B + 1, N1), dtype=torch.float64, device="cuda")
    joins = R.join_em(torch.from_numpy(S).cuda(), lo, hi, B, out)
    a = out.cpu().numpy()
    assert np.array_equal(joins, jref)
    fin = np.isfinite(ref)
    assert np.array_equal(np.isfinite(a), fin)
    assert np.max(np.abs(a[fin] - ref[fin])) <= 1e-11 * max(1.0, np.max(np.abs(ref[fin])))
    if h > 1:  # the last two windows share no point: refused
        S[h - 1, : hi[h - 2] - lo[h - 1] + 1] = -np.inf
        with pytest.raises(R.REWLError):
            R.join_em(torch.from_numpy(S).cuda(), lo, hi, B, out)
