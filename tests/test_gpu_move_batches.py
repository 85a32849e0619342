"""The move kernel's branches by size against the oracle, bit for bit: batches of 8, 16 and 32
steps (lattices on both sides of each limit), the three kinds of walk on both sides of the ln f
that separate them, non-dyadic and frozen windows, and replay with rows so wide
that the batch scratch does not fit beside them."""
import numpy as np
import pytest

import oracle as O
from tests import inputs as I
from tests.test_gpu_parity import FIELDS, _pair, _same, _replay_inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def cuda_lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_2328_gb300 import build as B
    B.build()


# lattices: 9 | 10 sites a side part batches of 8 and 16 steps, 21 | 22 those of 16 and 32
@pytest.mark.parametrize("model,L", [(0, 9), (0, 10), (3, 9), (10, 10), (0, 21), (0, 22), (10, 21),
                                     (7, 22)])
@pytest.mark.parametrize("lnf", [2.0 ** -5, 1.5 * 2.0 ** -6, 2.0 ** -7, 2.0 ** -8 * 1.01, 2.0 ** -12,
                                 2.0 ** -13, 3e-5, 2.0 ** -26])
def test_batch_sizes_and_walks_bit_exact(model, L, lnf):
    g, o = _pair(model, L, 2, 2, lnf_final=1e-9, seed=I.seed_for(7, L + model), interval=1777,
                 lnf_init=1.0)
    g.init()
    assert o.init() == 0
    g.run(max_rounds=2)  # ln g of some shape first
    o.run(2)
    g.set_state("lnf", np.full(2, lnf))
    o.put_window(lnf=np.full(2, lnf))
    g.run(max_rounds=3)
    o.run(3)
    g.set_state("finished", np.array([1, 0], np.uint8))  # window 0 frozen
    o.put_window(finished=np.array([1, 0], np.uint8))
    g.run(max_rounds=1)
    o.run(1)
    _same(g.state(), o.state(), FIELDS)
    g.close()


@pytest.mark.parametrize("call", ["replay", "replay_static"])
def test_replay_of_rows_that_fill_shared_memory(call):
    import paper_1402_2328_gb300.rewl as R
    model, L, n, T, W = 0, 4, 3, 70, 28500
    spins, k, lo, hi, lng, H, lnf, frozen, words = _replay_inputs(model, L, n, T, 12, 3, 0.8)
    wide = [np.zeros((n, W), a.dtype) for a in (lng, H)]
    for a, b in zip(wide, (lng, H)):
        a[:, :12] = b
    st = dict(spins=spins.copy(), k=k.copy(), lng=lng.copy(), H=H.copy())
    acc = np.zeros((n, T), np.int32)
    for t in range(T):
        r = O.replay_batch(model, 2, L, st["spins"], st["k"], lo, hi, st["lng"], st["H"], lnf,
                           frozen, words[:, t, :])
        st = dict(spins=r["spins"], k=r["k"], lng=r["lng"], H=r["H"])
        acc[:, t] = r["acc"]
    d = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a).view(dt)).cuda()  # noqa: E731
    sp, kd, lg, Hd = d(spins, np.int8), d(k, np.int32), d(wide[0], np.float64), d(wide[1], np.int32)
    ac, dk = (torch.zeros((n, T), dtype=torch.int32, device="cuda") for _ in range(2))
    getattr(R, call)(model, L, sp, kd, d(lo, np.int32), d(hi, np.int32), lg, Hd, d(lnf, np.float64),
                     d(frozen, np.uint8), d(words, np.int32), ac, dk)
    assert np.array_equal(ac.cpu().numpy(), acc)
    assert np.array_equal(sp.cpu().numpy(), st["spins"])
    assert np.array_equal(kd.cpu().numpy(), st["k"])
    assert np.array_equal(lg.cpu().numpy()[:, :12].view(np.uint64), st["lng"].view(np.uint64))
    assert np.array_equal(Hd.cpu().numpy().view(np.uint32)[:, :12], st["H"])


# windows narrower than one move's largest step, so that the prep walk can jump over them; a
# budget that ends inside a batch
@pytest.mark.parametrize("model,L,width,budget", [(0, 6, 3, 100), (3, 6, 3, 100), (10, 8, 2, 100),
                                                  (10, 13, 40, 1), (0, 13, 30, 1)])
def test_prep_bit_exact(model, L, width, budget):
    import paper_1402_2328_gb300.rewl as R
    B = O.num_bins(model, L)
    lo = np.arange(0, B - width + 1, max(1, width - 1), dtype=np.int32)
    hi = (lo + width).astype(np.int32)
    hi[-1] = B
    args = (model, L, len(lo), 0.75, 3, 1e-4, 0.8)
    seed = I.seed_for(8, L + model)
    g = R.REWL(model, L, 1, 0.75, 3, 1e-4, 0.8, seed=seed, prep_budget=budget)
    g.set_windows(lo, hi)
    o = O.REWL(*args, seed=seed, lo_hi=(lo, hi), prep_budget=budget)
    try:
        g.init()
        failed = False
    except R.REWLError:
        failed = True  # some window out of reach: the walkers' states still agree
    assert (o.init() != 0) == failed
    gs, os_ = {f: g.get_state(f) for f in ("spins", "k", "pstep", "prep_restarts")}, o.state()
    for f in gs:
        assert np.array_equal(gs[f], os_[f]), f
    g.close()


# more walkers than a second warp each fits the chip: one warp draws and walks
@pytest.mark.parametrize("model,L,h,m", [(0, 6, 2, 700), (10, 22, 4, 310)])
def test_many_walkers_bit_exact(model, L, h, m):
    g, o = _pair(model, L, h, m, seed=I.seed_for(9, L), interval=150)
    g.init()
    assert o.init() == 0
    g.run(max_rounds=2)
    o.run(2)
    g.set_state("lnf", np.full(h, 2.0 ** -12))
    o.put_window(lnf=np.full(h, 2.0 ** -12))
    g.run(max_rounds=1)
    o.run(1)
    _same(g.state(), o.state(), FIELDS)
    g.close()
