"""Lattices read back in slot order, in one copy to the host and in several (they go through 8 MB on the
device): what was written comes back, through a slot -> configuration map that exchanges have permuted,
and the call keeps no device memory of its own."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# 16-byte rows and odd ones; one copy, exactly full ones, and a remainder
@pytest.mark.parametrize("model,L,m", [(0, 32, 8), (2, 31, 5), (2, 128, 256), (0, 101, 409), (0, 101, 421)])
def test_lattices_come_back_in_slot_order(model, L, m):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_2328_gb300 import build as B
    B.build()
    import paper_1402_2328_gb300.rewl as R
    r = R.REWL(model, L, 4, 0.75, m, 1e-8, 0.8, seed=L, interval=50)
    r.init()
    r.run(max_rounds=8)
    assert r.get_state("swap_acc").sum() > 0
    free = torch.cuda.mem_get_info()[0]
    rng = np.random.default_rng(m)
    lat = rng.choice([-1, 1], (r.nw, r.N)) if model == 0 else rng.integers(0, model, (r.nw, r.N))
    r.set_state("spins", lat.astype(np.int8))
    assert np.array_equal(r.get_state("spins"), lat)
    assert free - torch.cuda.mem_get_info()[0] < 1 << 20
    r.close()
