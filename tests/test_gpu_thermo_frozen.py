"""Specific heat where one bin holds nearly all the weight and c is made of the rest, tens to hundreds of
orders of magnitude below N / T^2: every bin is then summed in float64, whether the float32 pass saw it
coming or the sum did.  Compared relatively, with everything taken relative to the bin of the largest
weight in numpy."""
import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _relative(lng, model, N, T):
    """c, and the weight of all bins but the largest one's relative to it."""
    E = -2.0 * N + (4.0 if model == 0 else 1.0) * np.arange(lng.size)
    E, l = E[np.isfinite(lng)], lng[np.isfinite(lng)]
    x = l - E / T
    i = np.argmax(x)
    w = np.exp((l - l[i]) - (E - E[i]) / T)
    d = (w * (E - E[i])).sum() / w.sum()
    return (w * (E - E[i] - d) ** 2).sum() / w.sum() / (N * T * T), np.delete(w, i).sum()


@pytest.mark.parametrize("model,L", [(0, 4), (3, 7), (10, 40), (0, 100)])
@pytest.mark.parametrize("shape", ["smooth", "holes", "rough"])
def test_specific_heat_of_a_frozen_lattice(model, L, shape):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_2328_gb300 import build as BB
    BB.build()
    import paper_1402_2328_gb300.rewl as R
    N, B = L * L, O.num_bins(model, L)
    k = np.arange(B + 1.0)
    lng = 0.7 * N * (1 - (2 * k / B - 1) ** 2)
    if shape == "holes":
        lng[1::3] = -np.inf
    elif shape == "rough":
        lng = lng + np.random.default_rng(L).normal(0, 3, B + 1)
    T = np.geomspace(0.008, 1.0, 400)
    ref = np.array([_relative(lng, model, N, t) for t in T])
    T, ref = T[ref[:, 0] > 1e-290], ref[ref[:, 0] > 1e-290]
    assert np.sum(ref[:, 1] < 1e-17) > 10 and np.sum((ref[:, 1] > 1e-17) & (ref[:, 1] < 1e-6)) > 5
    Td = torch.from_numpy(T).cuda()
    U, C = torch.zeros_like(Td), torch.zeros_like(Td)
    R.thermo(torch.from_numpy(lng).cuda(), model, L, Td, U, C)
    # an exponent, a difference of numbers up to |E/T| and |ln g|, has a few of their roundings; so does a
    # weight, relatively
    tol = 1e-12 + 8 * 2.0 ** -53 * (2 * N / T + np.max(np.abs(lng[np.isfinite(lng)])))
    assert np.all(np.abs(C.cpu().numpy() - ref[:, 0]) <= tol * ref[:, 0])
