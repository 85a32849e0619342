"""Joining against the oracle where the pairwise search has to start over: windows whose best join
bins do not come in order (noisy ln g), windows without a stencil, a single window, more windows than
one pass of shifts holds, and the jackknife of the same fragments."""
import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def cuda_lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_2328_gb300 import build as B
    B.build()


def _planted(model, L, lo, hi, m, seed, noise, holes):
    """Handles on both sides with every walker's ln g planted (rounds are not run)."""
    import paper_1402_2328_gb300.rewl as R
    h = len(lo)
    g = R.REWL(model, L, 1, 0.75, m, 1e-4, 0.8, seed=seed, interval=1)
    g.set_windows(lo, hi)
    o = O.REWL(model, L, h, 0.75, m, 1e-4, 0.8, seed=seed, interval=1, lo_hi=(lo, hi))
    try:
        g.init()
    except R.REWLError:
        pass  # walkers out of reach do not matter here
    o.init()
    rng = np.random.default_rng(seed)
    W, nw = g.W, h * m
    lng, mask = np.zeros((nw, W)), np.zeros((h, W), np.uint8)
    for w in range(h):
        nb = hi[w] - lo[w] + 1
        k = np.arange(lo[w], hi[w] + 1)
        mask[w, :nb] = rng.random(nb) >= holes
        mask[w, 0] = mask[w, nb - 1] = mask[w, nb // 2] = 1
        for i in range(m):
            lng[w * m + i, :nb] = (np.sqrt(k + 1.0) * 9 + rng.normal(0, noise, nb)) * mask[w, :nb]
    g.set_state("lng", lng)
    g.set_state("mask", mask)
    o.put(lng=lng)
    o.put_window(mask=mask)
    return g, o


@pytest.mark.parametrize("model,L,h,m,noise,holes", [
    (0, 8, 1, 2, 0.1, 0.0), (0, 8, 4, 3, 0.1, 0.0), (0, 16, 40, 2, 2.0, 0.0), (10, 12, 60, 2, 5.0, 0.3),
    (3, 9, 30, 1, 1.0, 0.7), (2, 8, 10, 2, 1.0, 0.0), (10, 30, 1100, 1, 0.5, 0.0)])
@pytest.mark.parametrize("norm", [0, 1])
def test_join_planted_windows(model, L, h, m, noise, holes, norm):
    B = O.num_bins(model, L)
    lo = (np.arange(h) * (B / (h + 3.0))).astype(np.int32)
    hi = np.minimum(B, lo + int(4 * B / (h + 3)) + 2).astype(np.int32)
    lo[0], hi[-1] = 0, B
    hi = np.maximum.accumulate(hi)
    keep = np.r_[True, (np.diff(hi) > 0) & (np.diff(lo) > 0)]
    lo, hi = lo[keep], hi[keep]
    hi[-1] = B
    g, o = _planted(model, L, lo, hi, m, 40 + L + h, noise, holes)
    try:
        a, ja = g.stitch(norm)
    except Exception:
        a = None
    try:
        b, jb = o.stitch(norm)
    except Exception:
        b = None
    assert (a is None) == (b is None)
    if a is None:
        return
    assert np.array_equal(ja, jb)
    fin = np.isfinite(b)
    assert np.array_equal(np.isfinite(a), fin)
    # sums of exponentials in another order: a few last bits of values up to a few thousand
    assert np.max(np.abs(a[fin] - b[fin])) < 1e-11
    g.close()
