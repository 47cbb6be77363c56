"""Kernel forms chosen by size give the same results: the small-system forms against the
large-system ones on the same structures (bit for bit where both keep the order of every sum).
"""
import numpy as np
import pytest

from paper_2205_10046_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_10046_gb300 import build
    build.build()
    return torch


def _dev(torch, pos, types):
    return torch.tensor(pos, device="cuda"), torch.tensor(types, device="cuda")


def _np(out):
    return {k: v.cpu().numpy() for k, v in out.items()}


def test_one_handle_serves_growing_and_shrinking_systems(torch_cuda):
    """The neighbour lists of a handle hold every system it is given next, also one with more
    atoms whose lists are no longer than the capacity that an earlier call settled on."""
    from paper_2205_10046_gb300 import nep
    torch = torch_cuda
    model = W.mixed_model(0)
    h = nep.NEP(model, skin=0.4)
    for n in (40, 500, 4001, 60000, 40, 4001):
        pos, types, box = W.random_structure(77, n)
        a = _np(h.compute(*_dev(torch, pos, types), box, per_atom_virial=True))
        fresh = nep.NEP(model, skin=0.4)
        b = _np(fresh.compute(*_dev(torch, pos, types), box, per_atom_virial=True))
        fresh.close()
        for k in ("U", "F", "W"):
            np.testing.assert_array_equal(a[k], b[k], err_msg=f"{k} of {n} atoms")
    h.close()
