"""Totals are plain FP64 sums of the per-atom values, infinities included: a chain of atoms whose
site energies and virials leave the FP32 range, among isolated atoms without either, at sizes on
both sides of the limits of the split kernels."""
import numpy as np
import pytest

from paper_2205_10046_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _huge(hyper):
    """Only f_0 enters, every neuron alike: U_i = n w1 tanh(0.1 q_0), W_i,xx = sum of positive terms, each
    below the FP32 range and their sum above it."""
    m = W.random_model(hyper, 0, [28.0] * hyper["n_types"])
    for a in (m.c_radial, m.c_angular, m.w0, m.b0, m.w1):
        a[...] = 0.0
    m.b1 = 0.0
    m.c_radial[:, :, 0, 0] = 1.0
    m.w0[:, 0] = 0.1
    m.w1[:] = 3.3e37 * 50 / hyper["n_neuron"]
    return m


GENERIC = dict(W.SI_MODEL, n_max_radial=5, basis_radial=5, n_neuron=50)


@pytest.mark.parametrize("hyper", [W.SI_MODEL, GENERIC], ids=["compiled", "runtime"])
@pytest.mark.parametrize("isolated", [0, 8000, 12000, 20000])
def test_infinite_terms_stay_infinite(torch_cuda, hyper, isolated):
    torch = torch_cuda
    from paper_2205_10046_gb300 import nep
    g = 7.0 * np.arange(29)
    grid = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    far = grid[grid[:, 2] >= 14.0][:isolated]  # nothing within 7 A of the chain or of each other
    chain = np.stack([np.arange(5.0), np.zeros(5), np.full(5, 1.0)], 1)
    pos = np.concatenate([chain, far])
    box = np.eye(3) * 7.0 * 31
    h = nep.NEP(_huge(hyper))
    out = h.compute(torch.tensor(pos, device="cuda"), torch.zeros(len(pos), dtype=torch.int32, device="cuda"), box,
                    per_atom_virial=True)
    o = {k: v.cpu().numpy() for k, v in out.items()}
    assert np.isposinf(o["U"]).any() and not np.isnan(o["U"]).any()
    assert np.isposinf(o["W"][:, 0]).any() and not np.isnan(o["W"]).any()
    assert np.isposinf(o["E"][0]) and np.isposinf(o["W_total"][0])
    np.testing.assert_array_equal(o["W_total"][1:], np.zeros(8))
    h.close()
