"""The run-time-shape kernels at the edges of their ranges, against the FP64 oracle: the largest
and the smallest model, more angular neighbours than one pass holds (16) and than a warp has
lanes, neurons just above a multiple of 32, atom counts around the 16 and 32 atoms of a block;
and a batch against its structures alone.

Bars as for the other run-time shapes: relative RMS 1e-5 for descriptors, energies, forces and
virials (FP32 sums of a few hundred terms, relative rounding 6e-8 each).
"""
import numpy as np
import pytest

import oracle
from paper_2205_10046_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# (types, rc_R, rc_A, n_R, n_A, K_R, K_A, l3b, l4b, l5b, neurons)
SHAPES = {
    "largest": (2, 6.0, 5.5, 19, 19, 19, 19, 4, 2, 1, 256),
    "smallest": (1, 4.0, 4.0, 0, 0, 0, 0, 1, 0, 0, 1),
    "four_body_on_l1": (3, 5.0, 3.0, 16, 7, 15, 11, 1, 2, 0, 33),
    "one_basis_apart": (1, 5.5, 5.5, 15, 3, 16, 16, 3, 2, 1, 31),
}


def _model(name):
    T, rcR, rcA, nR, nA, KR, KA, l3, l4, l5, H = SHAPES[name]
    hyper = dict(n_types=T, rc_radial=rcR, rc_angular=rcA, n_max_radial=nR, n_max_angular=nA, basis_radial=KR,
                 basis_angular=KA, l_max_3b=l3, l_max_4b=l4, l_max_5b=l5, n_neuron=H)
    return W.random_model(hyper, 7, [W.MASS_C, W.MASS_SI, W.MASS_GE][:T])


def _structures(name):
    return [W.random_structure(60 + n, n, n_types_model=SHAPES[name][0]) for n in (1, 15, 17, 33)]


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_10046_gb300 import build
    build.build()
    return torch


def _rel(a, b):
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-30)


@pytest.mark.parametrize("name", list(SHAPES))
def test_edges_match_oracle(torch_cuda, name):
    torch = torch_cuda
    from paper_2205_10046_gb300 import nep
    model = _model(name)
    h = nep.NEP(model)
    parts = _structures(name)
    alone = []
    for pos, types, box in parts:
        n = pos.shape[0]
        p, t = torch.tensor(pos, device="cuda"), torch.tensor(types, device="cuda")
        g = {k: v.cpu().numpy() for k, v in h.compute(p, t, box, per_atom_virial=True).items()}
        q = torch.zeros((n, model.n_des), dtype=torch.float64, device="cuda")
        nep.nep_descriptors(h.h, p, t, box, q)
        U, F, Wv = oracle.compute(model, pos, types, box)
        assert _rel(q.cpu().numpy(), oracle.descriptors(model, pos, types, box)) <= 1e-5
        assert _rel(g["U"], U) <= 1e-5
        # a lone atom's force is a sum of opposite image terms: compare with the largest term's scale
        scale = max(np.linalg.norm(F), 0.1 * np.linalg.norm(Wv))
        assert np.linalg.norm(g["F"] - F) <= 1e-5 * scale
        assert _rel(g["W"], Wv) <= 1e-5
        alone.append(g)
    b = W.concat_structures(parts)
    g = h.compute_batch(b.offsets, torch.tensor(b.pos, device="cuda"), torch.tensor(b.types, device="cuda"), b.boxes,
                        per_atom=True)
    g = {k: v.cpu().numpy() for k, v in g.items()}
    for s, one in enumerate(alone):
        a, e = int(b.offsets[s]), int(b.offsets[s + 1])
        for k in ("U", "F", "W"):
            np.testing.assert_array_equal(g[k][a:e], one[k], err_msg=f"{k} of {e - a} atoms")
    h.close()
