"""Canonical averages on the paths of k_thermo: smooth and bimodal ln g, unreachable bins, temperatures
where the float32 pass selects the bins and temperatures so low (or so extreme) that every bin is
taken in float64, against a float64 sum in numpy."""
import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _reference(lng, model, N, T):
    E = -2.0 * N + (4.0 if model == 0 else 1.0) * np.arange(lng.size)
    with np.errstate(all="ignore"):
        x = lng - E / T
        x = np.where(np.isfinite(lng), x, -np.inf)
        w = np.exp(x - x.max())
        u = (w * E).sum() / w.sum()
        c = (w * (E - u) ** 2).sum() / w.sum()
    return u / N, c / (N * T * T)


@pytest.mark.parametrize("model,L", [(0, 4), (3, 7), (10, 40), (0, 200)])
@pytest.mark.parametrize("shape", ["smooth", "holes", "two", "rough"])
def test_thermo_paths(model, L, shape):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_2328_gb300 import build as BB
    BB.build()
    import paper_1402_2328_gb300.rewl as R
    N, B = L * L, O.num_bins(model, L)
    k = np.arange(B + 1.0)
    lng = N * (1 - (2 * k / B - 1) ** 2)
    if shape == "holes":
        lng[1::3] = -np.inf
    elif shape == "two":
        lng = np.maximum(-((k - 0.2 * B) / 4) ** 2 + 10, -((k - 0.8 * B) / (0.05 * B + 2)) ** 2)
    elif shape == "rough":
        lng = lng + np.random.default_rng(L).normal(0, 20, B + 1)
    T = np.array([1e-6, 1e-3, 0.05, 0.4, 1.0, 2.27, 30.0, 1e6, -1.5, np.inf])
    Td = torch.from_numpy(T).cuda()
    U, C = torch.zeros_like(Td), torch.zeros_like(Td)
    R.thermo(torch.from_numpy(lng).cuda(), model, L, Td, U, C)
    U, C = U.cpu().numpy(), C.cpu().numpy()
    for i, t in enumerate(T):
        u, c = _reference(lng, model, N, t)
        # quotients and exponents of up to |E/T|: their rounding, times a few
        tol = 1e-12 + 1e-15 * (2 * N / abs(t) + np.max(np.abs(lng[np.isfinite(lng)])))
        assert abs(U[i] - u) <= tol * max(1.0, abs(u)), (t, U[i], u)
        assert abs(C[i] - c) <= tol * max(abs(c), N / (t * t) * 1e-3, 1e-300) or abs(C[i] - c) <= 1e-9 * abs(c), \
            (t, C[i], c)
