"""Calls of different kinds on one handle: a batch whose layout repeats after a single structure
was evaluated, simulated or described in between gives the same bits as before, on the eager path
and when the captured graph would replay."""
import numpy as np
import pytest

from paper_2205_10046_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("between", ["compute", "descriptors", "md_init", "heat_current", "refused_box"])
@pytest.mark.parametrize("calls_before", [1, 3])  # 3: the batch graph is captured
@pytest.mark.parametrize("sizes", [[40, 8, 300, 77], [9]])
def test_batch_layout_after_a_single_structure(torch_cuda, sizes, calls_before, between):
    torch = torch_cuda
    from paper_2205_10046_gb300 import nep
    model = W.mixed_model(0)
    b = W.concat_structures([W.random_structure(50 + k, n) for k, n in enumerate(sizes)])
    dev = lambda a, dt=torch.float64: torch.tensor(a, dtype=dt, device="cuda")  # noqa: E731
    p, t = dev(b.pos), dev(b.types, torch.int32)
    # another box, image range and atom count, fewer and more cells than the batch
    singles = [W.random_structure(60, 12), W.random_structure(61, 2500)]
    out = {k: dev(np.zeros(s)) for k, s in dict(U=b.n_atoms, E=b.n_struct, F=(b.n_atoms, 3), W=(b.n_atoms, 9),
                                                Ws=(b.n_struct, 9)).items()}

    def batch(h):
        nep.nep_compute_batch(h.h, b.offsets, p, t, b.boxes, out["U"], out["E"], out["F"], out["W"], out["Ws"])
        return {k: v.cpu().numpy().copy() for k, v in out.items()}

    z = dev(np.stack([model.to_vector(), W.mixed_model(3).to_vector()]))
    targets = [dev(np.full(s, 0.1)) for s in (b.n_struct, (b.n_atoms, 3), (b.n_struct, 6))]

    def population(h):
        return nep.nep_eval_population(h.h, z, b.offsets, p, t, b.boxes, *targets).cpu().numpy()

    fresh = nep.NEP(model, skin=0.4)
    ref_pop = population(fresh)
    fresh.close()
    h = nep.NEP(model, skin=0.4)
    ref = batch(h)
    for _ in range(calls_before - 1):
        batch(h)
    assert (nep.nep_get_stats(h.h)["batch_graph_kernels"] > 0) == (calls_before > 1)
    for pos, types, box in singles:
        sp, st, n = dev(pos), dev(types, torch.int32), len(types)
        if between == "compute":
            h.compute(sp, st, box)
        elif between == "descriptors":
            nep.nep_descriptors(h.h, sp, st, box, dev(np.zeros((n, nep.nep_n_des(h.h)))))
        elif between == "md_init":
            nep.md_init(h.h, sp, st, box)
            nep.md_run(h.h, 2, 1.0)
        elif between == "heat_current":
            nep.nep_heat_current(h.h, sp, st, box, dev(np.ones((n, 3))), None, dev(np.zeros(3)))
        else:
            with pytest.raises(nep.NepError):
                h.compute(sp, st, np.diag([0.5, 20.0, 20.0]))
        for _ in range(2):
            got = batch(h)
            for k in ref:
                np.testing.assert_array_equal(got[k], ref[k], err_msg=k)
        lists = nep.nep_export_lists(h.h, b.n_atoms)  # of the batch, in its own packing
        for s in range(b.n_struct):
            a, e = b.offsets[s], b.offsets[s + 1]
            j = np.concatenate([lists["j_r"][i, :lists["nn_r"][i]] for i in range(a, e)])
            assert j.min() >= a and j.max() < e
        np.testing.assert_array_equal(population(h), ref_pop)
    h.close()
