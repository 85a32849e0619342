"""The gradient kernel at the edges of its tiles (two CTAs of 64 samples each): fewer samples than one
CTA, exactly one, one more, a tile and one more; training steps equal gradient and Adam calls."""
import numpy as np
import pytest

from oracle import mlp as M
from tests import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_2328_gb300 import build as B
    B.build()
    import paper_1402_2328_gb300.rewl as R
    return R


@pytest.mark.parametrize("n", [1, 63, 64, 65, 127, 128, 129, 300])
def test_gradient_at_tile_edges(R, n):
    p = I.mlp_params(8, scale=0.15)
    X, T = I.mlp_data(9, n)
    P = torch.tensor(p, dtype=torch.float32, device="cuda")
    Xd, Td = torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda()
    grad = torch.zeros(M.NPARAM, device="cuda")
    loss = torch.zeros(1, device="cuda")
    work = torch.full((R.mlp_workspace_floats(n),), float("nan"), device="cuda")
    R.mlp_grad(P, Xd, Td, grad, loss, work)
    l_ref, g_ref = M.loss_and_grad(p, X, T)
    # float32 against float64: 24-bit mantissa, sums of at most 64 + n terms
    assert loss.item() == pytest.approx(l_ref, rel=1e-4)
    assert np.max(np.abs(grad.cpu().numpy() - g_ref)) < 1e-4 * np.max(np.abs(g_ref))
    # training = gradient + Adam, bit for bit
    a, b = P.clone(), P.clone()
    ma, va, mb, vb = (torch.zeros_like(P) for _ in range(4))
    ga, gb = torch.zeros_like(P), torch.zeros_like(P)
    R.mlp_train(a, Xd, Td, 3, 1e-3, 4, ma, va, ga, work, loss)
    for t in (5, 6, 7):
        R.mlp_grad(b, Xd, Td, gb, loss, work)
        R.mlp_adam(b, gb, mb, vb, t, 1e-3)
    for x, y in ((a, b), (ma, mb), (va, vb), (ga, gb)):
        assert torch.equal(x, y)
