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


@pytest.mark.parametrize("name", ["si", "pbte", "mixed"])
def test_split_forms_equal_the_plain_ones(torch_cuda, name):
    """Small systems share an atom's work among four or two groups of lanes (kernel limits 7,296,
    9,728, 14,592 and 19,456 atoms); a batch of all of them together does not. The same bits per
    atom, and totals that are their sums (pairs of FP32 words, about 48 bits: 1e-9 is ample)."""
    from paper_2205_10046_gb300 import nep
    torch = torch_cuda
    model = {"si": lambda: W.random_model(W.SI_MODEL, 0, [W.MASS_SI]),
             "pbte": lambda: W.random_model(W.PBTE_MODEL, 1, [W.MASS_PB, W.MASS_TE]),
             "mixed": lambda: W.mixed_model(0)}[name]()
    sizes = [1, 16, 33, 7296, 7297, 9729, 14592, 14593, 19457]
    parts = [W.random_structure(700 + k, n, n_types_model=model.n_types) for k, n in enumerate(sizes)]
    b = W.concat_structures(parts)
    h = nep.NEP(model, skin=0.4)
    g = _np(h.compute_batch(b.offsets, *_dev(torch, b.pos, b.types), b.boxes, per_atom=True))
    for s in range(b.n_struct):
        pos, types, box = b.structure(s)
        a, e = int(b.offsets[s]), int(b.offsets[s + 1])
        dev = _dev(torch, pos, types)
        one = _np(h.compute(*dev, box, per_atom_virial=True))
        few = _np(h.compute_batch(np.array([0, e - a]), *dev, np.asarray(box).reshape(1, 9), per_atom=True))
        for k in ("U", "F", "W"):
            np.testing.assert_array_equal(g[k][a:e], one[k], err_msg=f"{k} of {e - a} atoms")
            np.testing.assert_array_equal(g[k][a:e], few[k], err_msg=f"{k} of {e - a} atoms, batch of one")
        assert abs(one["E"][0] - one["U"].sum()) <= 1e-9 * np.abs(one["U"]).sum()
        assert np.abs(one["W_total"].reshape(9) - one["W"].sum(0)).max() <= 1e-9 * np.abs(one["W"]).sum()
    h.close()
