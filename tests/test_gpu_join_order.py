"""The jackknife's many joins at once, in several passes over the resamples, against the oracle."""
import numpy as np
import pytest

import oracle as O
from tests.test_gpu_join import cuda_lib  # noqa: F401 (fixture)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


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
