"""The second warp of a walker draws its proposals into a ring of 128 steps, 32 at a time, and the first
takes them in batches of at most 32: launches shorter than a block, as long as one, the ring and both with
a step more or less, on both models and in all three forms of the walk, against the oracle bit for bit.
(The kernels with every decision checked in float64 as well draw in the walking warp.)"""
import numpy as np
import pytest

from tests import inputs as I
from tests.test_gpu_parity import FIELDS, _pair, _same

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def cuda_lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_2328_gb300 import build as B
    B.build()


@pytest.mark.parametrize("model,L", [(0, 8), (10, 12), (0, 24), (10, 24)])
@pytest.mark.parametrize("lnf", [1.0, 2.0 ** -8, 2.0 ** -18])
def test_launch_lengths_around_block_and_ring(model, L, lnf):
    for interval in (1, 31, 32, 33, 63, 64, 65, 95, 96, 97, 127, 128, 129, 160, 161, 1000):
        g, o = _pair(model, L, 2, 3, lnf_final=1e-9, seed=I.seed_for(11, interval), interval=interval)
        g.init()
        assert o.init() == 0
        g.set_state("lnf", np.full(2, lnf))
        o.put_window(lnf=np.full(2, lnf))
        g.run(max_rounds=6)
        o.run(6)
        _same(g.state(), o.state(), FIELDS)
        g.close()


# The start bin counts as visited from the first batch on: a launch that saw it as not visited would send
# the steps from and to it to the float64 path.  The path taken, not only its result, is a function of the
# state, so every repetition of a run counts the same number of float64 decisions.
@pytest.mark.parametrize("model,L", [(0, 16), (10, 16)])
def test_start_bin_is_visited_in_every_launch(model, L):
    import paper_1402_2328_gb300.rewl as R
    counts = []
    for _ in range(4):
        r = R.REWL(model, L, 4, 0.75, 8, 1e-9, 0.8, seed=I.seed_for(12, L), interval=200)
        r.init()
        r.run(max_rounds=50)
        r.set_state("mask", np.zeros((r.h, r.W), np.uint8))  # only the start bin of each launch
        r.set_state("lnf", np.full(4, 2.0 ** -16))
        r.run(max_rounds=1)
        counts.append(int(r.get_state("n_exact")[0]))
        r.close()
    assert len(set(counts)) == 1, counts
