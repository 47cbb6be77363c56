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


def test_large_batch_equals_its_structures_alone(torch_cuda):
    """A batch of more than 131,072 atoms takes the large-system forms of the list build and of
    the force kernels, its structures alone the small-system ones: the same lists in the same
    order and the same forces, bit for bit. Sizes: tiny cells (several images per axis), ragged
    and odd counts, one structure just above a warp and one that makes up the bulk."""
    from paper_2205_10046_gb300 import nep
    torch = torch_cuda
    sizes = [8, 31, 33, 127, 500, 4001, 0, 131072]
    parts = [W.random_structure(9000 + k, n) if n else (np.zeros((0, 3)), np.zeros(0, np.int32), np.eye(3) * 9.0)
             for k, n in enumerate(sizes)]
    b = W.concat_structures(parts)
    assert b.n_atoms > 131072
    model = W.mixed_model(0)
    h = nep.NEP(model, skin=0.4)
    p, t = _dev(torch, b.pos, b.types)
    g = _np(h.compute_batch(b.offsets, p, t, b.boxes, per_atom=True))
    st = nep.nep_get_stats(h.h)
    cap = max(st["max_radial"], st["max_angular"])
    lists = nep.nep_export_lists(h.h, b.n_atoms, cap)
    h1 = nep.NEP(model, skin=0.4)
    for s in range(b.n_struct):
        pos, types, box = b.structure(s)
        if pos.shape[0] == 0:
            continue
        a, e = int(b.offsets[s]), int(b.offsets[s + 1])
        one = _np(h1.compute(*_dev(torch, pos, types), box, per_atom_virial=True))
        for k in ("U", "F", "W"):
            np.testing.assert_array_equal(g[k][a:e], one[k], err_msg=f"{k} of {e - a} atoms")
        l1 = nep.nep_export_lists(h1.h, e - a, cap)
        for r, nn in (("r", "nn_r"), ("a", "nn_a")):
            np.testing.assert_array_equal(lists[nn][a:e], l1[nn])
            m = np.arange(cap)[None, :] < l1[nn][:, None]
            np.testing.assert_array_equal(lists["j_" + r][a:e][m] - a, l1["j_" + r][m])
            np.testing.assert_array_equal(lists["d_" + r][a:e][m], l1["d_" + r][m])
    h.close()
    h1.close()
