"""Positions and types outside the GPU's own memory (page-locked host arrays here; another GPU's memory
takes the same way) give the bits of device arrays through every call that takes a structure."""
import ctypes as C

import numpy as np
import pytest

from paper_2205_10046_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [300, 140000])  # the one-kernel build and the separate kernels
def test_inputs_in_host_memory(torch_cuda, n):
    torch = torch_cuda
    from paper_2205_10046_gb300 import nep
    lib = nep.load()
    model = W.mixed_model(0)
    parts = [W.random_structure(90 + k, m) for k, m in enumerate((n // 3, n - n // 3))]
    b = W.concat_structures(parts)
    pos, types, box = W.random_structure(95, n)
    box = np.ascontiguousarray(box)
    off, boxes = np.ascontiguousarray(b.offsets, np.int32), np.ascontiguousarray(b.boxes, np.float64)
    cur = torch.cuda.current_stream().cuda_stream
    new = lambda *s: torch.zeros(s, dtype=torch.float64, device="cuda")  # noqa: E731
    p, _keep = nep._params(model, 0.4)
    targets = [new(2), new(n, 3)]
    lam = np.array([1.0, 1.0, 0.0, 0.0, 0.0])
    z = torch.tensor(model.to_vector()[None], device="cuda")

    def calls(place):
        put = lambda a: place(torch.tensor(a))  # noqa: E731
        sp, st, bp, bt = put(pos), put(types.astype(np.int32)), put(b.pos), put(b.types.astype(np.int32))
        h = nep.NEP(model, skin=0.4)
        out = []

        def call(f, *outputs):
            assert f() == 0, lib.nep_last_error(h.h)
            torch.cuda.synchronize()
            out.extend(o.cpu().numpy().copy() for o in outputs)

        E, F, Wt = new(1), new(n, 3), new(9)
        call(lambda: lib.nep_compute(h.h, n, sp.data_ptr(), st.data_ptr(), box.ctypes.data, None, E.data_ptr(),
                                     F.data_ptr(), None, Wt.data_ptr(), cur), E, F, Wt)
        x = new(n, 3)
        call(lambda: lib.md_init(h.h, n, sp.data_ptr(), st.data_ptr(), box.ctypes.data, None, cur))
        call(lambda: lib.md_run(h.h, 2, 1.0, 1, None, cur))
        call(lambda: lib.md_get_state(h.h, x.data_ptr(), None, None, cur), x)
        Es, Fb = new(2), new(n, 3)
        for _ in range(4):  # eager, captured, replayed
            call(lambda: lib.nep_compute_batch(h.h, 2, off.ctypes.data, bp.data_ptr(), bt.data_ptr(), boxes.ctypes.data,
                                               None, Es.data_ptr(), Fb.data_ptr(), None, None, cur), Es, Fb)
        assert nep.nep_get_stats(h.h)["batch_graph_kernels"] > 0
        loss = new(1, 6)
        call(lambda: lib.nep_eval_population(h.h, 1, z.data_ptr(), 2, off.ctypes.data, bp.data_ptr(), bt.data_ptr(),
                                             boxes.ctypes.data, targets[0].data_ptr(), targets[1].data_ptr(), None,
                                             lam.ctypes.data, loss.data_ptr(), cur), loss)
        if n <= 4096:
            q = new(n, model.n_des)
            call(lambda: lib.nep_descriptors_static(C.byref(p), n, sp.data_ptr(), st.data_ptr(), box.ctypes.data,
                                                    q.data_ptr(), cur), q)
        h.close()
        return out

    for a, r in zip(calls(lambda t: t.pin_memory()), calls(lambda t: t.cuda())):
        np.testing.assert_array_equal(a, r)
