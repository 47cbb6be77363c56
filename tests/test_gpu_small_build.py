"""The one-kernel neighbour build alone and over batches: sizes around its blocks, a grid with more
cells than atoms on both sides of the 8,192 cells where its prefix sum changes, atoms outside the
cell, batches, and inputs it has to refuse."""
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


def _outside(pos, box, seed):
    """Some of the atoms moved by whole cell vectors."""
    k = np.random.default_rng(seed).integers(-2, 3, size=pos.shape) * (np.arange(pos.shape[0]) % 3 == 0)[:, None]
    return pos + k @ np.asarray(box).reshape(3, 3)


@pytest.mark.parametrize("sizes", [[1, 2, 1023, 1024, 1025], [2047, 2048, 2049], [7] * 290, "dilute"])
def test_structure_alone_equals_batch(torch_cuda, sizes):
    """A structure alone and in a batch, split over the blocks in other places: the same atom order,
    lists and sums, hence the same bits."""
    from paper_2205_10046_gb300 import nep
    torch = torch_cuda
    if sizes == "dilute":  # more cells than atoms: 4 per atom at most, 8,192 and more in all
        rng = np.random.default_rng(5)
        parts = [(rng.random((n, 3)) * 400.0, rng.integers(0, W.mixed_model(0).n_types, n).astype(np.int32), np.eye(3) * 400.0)
                 for n in (1900, 2048, 300)]
    else:
        parts = [W.random_structure(400 + k, n) for k, n in enumerate(sizes)]
    parts = [(_outside(p, box, k), t, box) for k, (p, t, box) in enumerate(parts)]
    b = W.concat_structures(parts)
    model = W.mixed_model(0)
    h, h1 = nep.NEP(model, skin=0.4), nep.NEP(model, skin=0.4)
    g = _np(h.compute_batch(b.offsets, *_dev(torch, b.pos, b.types), b.boxes, per_atom=True))
    for s in list(range(b.n_struct))[:12]:
        pos, types, box = b.structure(s)
        a, e = int(b.offsets[s]), int(b.offsets[s + 1])
        one = _np(h1.compute(*_dev(torch, pos, types), box, per_atom_virial=True))
        for k in ("U", "F", "W"):
            np.testing.assert_array_equal(g[k][a:e], one[k], err_msg=f"{k} of {e - a} atoms")
    h.close()
    h1.close()


@pytest.mark.parametrize("n", [300, 3000])
def test_outputs_untouched_by_refused_input(torch_cuda, n):
    """Kernels queued behind a build that fails write nothing, and the next call is right; lists
    that outgrow their capacity are built again."""
    from paper_2205_10046_gb300 import nep
    torch = torch_cuda
    model = W.mixed_model(0)
    pos, types, box = W.random_structure(31, n)
    h = nep.NEP(model, skin=0.4)
    wide = _np(h.compute(*_dev(torch, pos * 3.0, types), np.asarray(box) * 3.0, per_atom_virial=True))  # short lists
    got = _np(h.compute(*_dev(torch, pos, types), box, per_atom_virial=True))
    fresh = nep.NEP(model, skin=0.4)
    ref = _np(fresh.compute(*_dev(torch, pos, types), box, per_atom_virial=True))
    for k in ("U", "F", "W", "E", "W_total"):
        np.testing.assert_array_equal(got[k], ref[k])
    outs = [torch.full((m,), 7.0, dtype=torch.float64, device="cuda") for m in (n, 1, 3 * n, 9 * n, 9)]
    for what in ("type", "nan"):
        p, t = _dev(torch, pos, types)
        if what == "type":
            t[n - 1] = 9
        else:
            p[n // 2, 1] = float("nan")
        with pytest.raises(nep.NepError):
            nep.nep_compute(h.h, p, t, box, outs[0], outs[1], outs[2].view(n, 3), outs[3].view(n, 9), outs[4])
        torch.cuda.synchronize()
        assert all(bool((o == 7.0).all()) for o in outs)
    again = _np(h.compute(*_dev(torch, pos * 3.0, types), np.asarray(box) * 3.0, per_atom_virial=True))
    for k in ("U", "F", "W", "E", "W_total"):
        np.testing.assert_array_equal(again[k], wide[k])
    h.close()
    fresh.close()
