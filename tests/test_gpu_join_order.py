"""Joining where a pair's best bin is not the answer: bins out of order (the pair is searched again behind
the join before it), overlaps with only a 3-point stencil or none, and the jackknife's many joins at
once, in one pass over the resamples and in several, against the oracle.  Each case says what it is
meant to reach, and an independent search checks that it does."""
import numpy as np
import pytest

import oracle as O
from tests.test_gpu_join import _planted, cuda_lib  # noqa: F401 (fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _beta(l, v, b, npts, step, de):
    at = [b - step, b + step] + ([b - 2 * step, b + 2 * step] if npts == 5 else [])
    if min(at) < 0 or max(at) >= len(l) or not all(v[i] for i in at):
        return None
    if npts == 5:
        return ((8 * l[b + step] - l[b + 2 * step]) - 8 * l[b - step] + l[b - 2 * step]) / (12 * de * step)
    return (l[b + step] - l[b - step]) / (2 * de * step)


def _best_alone(model, lo, hi, mean, mask):
    """Join bin of every pair as if it were alone, and the stencil that found it (5, 3, 0: none)."""
    de, step = (4.0 if model == 0 else 1.0), (2 if model == 2 else 1)
    bins, kinds = [], []
    for w in range(len(lo) - 1):
        win = [(mean[i][: hi[i] - lo[i] + 1], mask[i][: hi[i] - lo[i] + 1], lo[i]) for i in (w, w + 1)]
        ks = [k for k in range(lo[w + 1], hi[w] + 1) if all(v[k - a] for _, v, a in win)]
        for npts in (5, 3, 0):
            if npts:
                at = [(k, [_beta(l, v, k - a, npts, step, de) for l, v, a in win]) for k in ks]
                c = [(abs(b[0] - b[1]), k) for k, b in at if None not in b]
            else:
                c = [(abs(2 * k - (lo[w + 1] + hi[w])), k) for k in ks]
            if c:
                bins.append(min(c)[1])
                kinds.append(npts)
                break
    return bins, kinds


def _out_of_order(bins):
    return sum(b <= a for a, b in zip(bins, bins[1:]))


# window i overlaps i + 1 in ten bins and no other window, so each pair's stencil is planted by itself:
# visited runs of three bins leave only the 3-point one, single bins none
@pytest.mark.parametrize("model,m", [(0, 1), (3, 2)])
@pytest.mark.parametrize("norm", [0, 1])
def test_stencils_of_each_pair(model, m, norm):
    L = 17 if model == 0 else 12
    B = O.num_bins(model, L)
    lo = (21 * np.arange(B // 21 - 1)).astype(np.int32)
    hi = lo + 30
    hi[-1] = B
    g, o = _planted(model, L, lo, hi, m, 77 + model, 0.3, 0.0)
    mask = o.state()["mask"].copy()
    want = [(5, 3, 0)[w % 3] for w in range(len(lo) - 1)]
    for w, kind in enumerate(want):
        for k in range(lo[w + 1], hi[w] + 1):
            seen = kind == 5 or (kind == 3 and (k - lo[w + 1]) % 4 < 3) or (kind == 0 and (k - lo[w + 1]) % 2 == 0)
            mask[w, k - lo[w]] = mask[w + 1, k - lo[w + 1]] = seen
    g.set_state("mask", mask)
    o.put_window(mask=mask)
    mean = [o.window_mean(w) for w in range(len(lo))]
    assert _best_alone(model, lo, hi, mean, mask)[1] == want
    a, ja = g.stitch(norm)
    b, jb = o.stitch(norm)
    assert np.array_equal(ja, jb)
    fin = np.isfinite(b)
    assert np.array_equal(np.isfinite(a), fin)
    # sums of exponentials in another order: a few last bits of values up to a few thousand
    assert np.max(np.abs(a[fin] - b[fin])) < 1e-11
    g.close()


# on both sides of the limits up to which one CTA searches all pairs: 2 windows whatever their size, 8
# windows, 192 bins
@pytest.mark.parametrize("h,W", [(2, 900), (8, 192), (8, 193), (9, 150)])
def test_pairs_searched_by_one_cta_and_by_many(h, W):
    model, L = 0, 32
    B = O.num_bins(model, L)
    lo = ((B - W + 1) * np.arange(h) // (h - 1)).astype(np.int32)
    hi = (lo + W - 1).astype(np.int32)
    g, o = _planted(model, L, lo, hi, 2, 90 + h + W, 3.0, 0.0)
    assert (g.h, g.W) == (h, W)
    a, ja = g.stitch()
    b, jb = o.stitch()
    assert np.array_equal(ja, jb)
    assert np.array_equal(np.isfinite(a), np.isfinite(b))
    fin = np.isfinite(b)
    assert np.max(np.abs(a[fin] - b[fin])) < 1e-11  # as above
    g.close()


def _finished_pair(model, L, h, m, interval, seed, lnf_final=2.0 ** -3):
    """Short runs taken through all their iterations (every check counts as flat): noisy fragments."""
    import paper_1402_2328_gb300.rewl as R
    args = (model, L, h, 0.75, m, lnf_final, 0.0)
    g, o = R.REWL(*args, seed=seed, interval=interval), O.REWL(*args, seed=seed, interval=interval)
    g.init()
    assert o.init() == 0
    g.run(max_rounds=40)
    o.run(40)
    a, b = g.state(), o.state()
    assert np.all(b["finished"] == 1)
    assert np.array_equal(a["frag"], b["frag"]) and np.array_equal(a["mask"], b["mask"])
    return g, o


def _same_error(g, o, norm):
    a, b = g.jackknife(norm), o.jackknife(norm)
    assert np.array_equal(np.isnan(a), np.isnan(b))
    fin = ~np.isnan(b)
    # m resamples of values of at most `big`: a few roundings each, the mean's m of them, and the root of
    # a sum of m squares of such differences
    big = np.max(np.abs(o.state()["frag"])) * o.h + o.N * np.log(o.q)
    tol = 4 * g.m ** 1.5 * 2.0 ** -53 * big
    assert np.max(np.abs(a[fin] - b[fin])) <= tol
    assert np.max(b[fin]) > 1e3 * tol  # and the error is something


# pairs searched again in some resamples, fewer and more windows than are joined by one CTA alone; model 2
# has stencils of step 2
@pytest.mark.parametrize("model,L,h,m,interval,seed", [
    (0, 8, 6, 3, 400, 1), (0, 12, 8, 5, 800, 7), (2, 8, 6, 3, 600, 9), (3, 8, 12, 2, 800, 6),
    (0, 16, 12, 4, 1500, 4), (10, 10, 20, 3, 1500, 5), (0, 16, 40, 2, 2000, 8)])
@pytest.mark.parametrize("norm", [0, 1])
def test_jackknife_with_bins_out_of_order(model, L, h, m, interval, seed, norm):
    g, o = _finished_pair(model, L, h, m, interval, seed)
    s = o.state()
    frag = s["frag"].reshape(h, m, -1)
    again = [_out_of_order(_best_alone(model, o.lo, o.hi, (frag.sum(1) - frag[:, j]) / (m - 1), s["mask"])[0])
             for j in range(m)]
    assert max(again) > 0  # searched again in some resample
    _same_error(g, o, norm)
    g.close()


# 1024 resamples take more than the workspace that a handle keeps: several passes, with the resamples'
# results beside the workspace and (the larger lattice) in an allocation of the call
@pytest.mark.parametrize("model,L,h,interval", [(0, 32, 4, 2000), (3, 33, 2, 1500)])
def test_jackknife_in_several_passes_keeps_a_bounded_workspace(model, L, h, interval):
    g, o = _finished_pair(model, L, h, 1024, interval, 21, 2.0 ** -5)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    _same_error(g, o, 0)
    kept = free - torch.cuda.mem_get_info()[0]
    assert kept <= (16 << 20) + (2 << 20)  # 16 MB, in the allocator's pages
    first = g.jackknife()
    assert np.array_equal(first, g.jackknife(), equal_nan=True)
    g.close()
