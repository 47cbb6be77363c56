"""Waits of the one-kernel neighbour build that run out (a limit of one poll): the call ends with
NEP_ERR_TIMEOUT, nothing is written to its outputs, and the next call with the usual limit is right."""
import numpy as np
import pytest

from paper_2205_10046_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TIMEOUT, STATE = -8, -7


def _raises(code, f):
    from paper_2205_10046_gb300 import nep
    with pytest.raises(nep.NepError) as e:
        f()
    assert e.value.code == code
    if code == TIMEOUT:
        assert "barrier of the neighbour build" in str(e.value)


@pytest.mark.parametrize("n", [300, 20000])
@pytest.mark.parametrize("first", [True, False])  # on a handle without and with lists
def test_calls_end_with_the_wait(torch_cuda, n, first):
    torch = torch_cuda
    from paper_2205_10046_gb300 import nep
    model = W.mixed_model(0)
    pos, types, box = W.random_structure(21, n)
    p, t = torch.tensor(pos, device="cuda"), torch.tensor(types, device="cuda")
    out = [torch.full(s, 7.0, dtype=torch.float64, device="cuda") for s in ((n,), (1,), (n, 3), (n, 9), (9,))]
    off, boxes = np.array([0, n // 3, n], np.int32), np.stack([box, box])
    ws = [torch.full(s, 7.0, dtype=torch.float64, device="cuda") for s in ((2,), (2, 9))]
    single = lambda h: nep.nep_compute(h.h, p, t, box, *out)  # noqa: E731
    batch = lambda h: nep.nep_compute_batch(h.h, off, p, t, boxes, out[0], ws[0], out[2], out[3], ws[1])  # noqa: E731
    for call in (single, batch):
        h, ref = nep.NEP(model, skin=0.4), nep.NEP(model, skin=0.4)
        if not first:
            call(h)
        for o in out + ws:
            o.fill_(7.0)
        nep.nep_set_wait_limit(h.h, 1)
        for _ in range(2):
            _raises(TIMEOUT, lambda: call(h))
            torch.cuda.synchronize()
            assert all(bool((o == 7.0).all()) for o in out + ws)
        _raises(STATE, lambda: nep.nep_export_lists(h.h, n, 4))
        nep.nep_set_wait_limit(h.h, 0)
        for _ in range(3):
            call(h)
        got = [o.cpu().numpy().copy() for o in out + ws]
        call(ref)
        for a, o in zip(got, out + ws):
            np.testing.assert_array_equal(a, o.cpu().numpy())
        h.close()
        ref.close()


def _hot(torch, w):
    """Velocities that move every atom past skin/2 in the first step of 1 fs."""
    v = torch.randn((w.n_atoms, 3), dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(4))
    return 0.3 * v / v.norm(dim=1, keepdim=True)


@pytest.mark.parametrize("reps", [3, 12])  # 216 and 13,824 atoms
def test_md_ends_with_the_wait(torch_cuda, reps):
    torch = torch_cuda
    from paper_2205_10046_gb300 import nep
    w = W.si_diamond(reps, seed=4)
    pos, types, vel = torch.tensor(w.pos, device="cuda"), torch.tensor(w.types, device="cuda"), _hot(torch, w)
    h, ref = nep.NEP(w.model, skin=0.4), nep.NEP(w.model, skin=0.4)
    x, xr = torch.empty_like(pos), torch.empty_like(pos)

    def run(hh, out):
        nep.md_init(hh.h, pos, types, w.box, vel)
        nep.md_run(hh.h, 4, 1.0)
        nep.md_get_state(hh.h, pos=out)

    run(ref, xr)
    for steps in (lambda: nep.md_run(h.h, 4, 1.0), lambda: (nep.md_run_async(h.h, 4, 1.0), nep.md_status(h.h)),
                  lambda: nep.fire_run(h.h, 4, 300.0, 0.0)):
        nep.md_init(h.h, pos, types, w.box, vel)
        nep.nep_set_wait_limit(h.h, 1)
        _raises(TIMEOUT, steps)
        _raises(STATE, lambda: nep.md_get_state(h.h, pos=x))
        _raises(TIMEOUT, lambda: nep.md_init(h.h, pos, types, w.box, vel))
        nep.nep_set_wait_limit(h.h, 0)
        run(h, x)
        np.testing.assert_array_equal(x.cpu().numpy(), xr.cpu().numpy())
    ref.close()
    h.close()


@pytest.mark.parametrize("reps", [3, 12])
@pytest.mark.parametrize("next_call", ["compute", "md", "batch", "stats"])
def test_calls_after_an_unseen_time_out(torch_cuda, reps, next_call):
    """The build of a step queued by md_run_async runs out and no call asks for it: the next one
    starts from a cleared barrier all the same."""
    torch = torch_cuda
    from paper_2205_10046_gb300 import nep
    w = W.si_diamond(reps, seed=6)
    pos, types, vel = torch.tensor(w.pos, device="cuda"), torch.tensor(w.types, device="cuda"), _hot(torch, w)
    off, boxes = np.array([0, w.n_atoms], np.int32), np.asarray(w.box)[None]
    h, ref = nep.NEP(w.model, skin=0.4), nep.NEP(w.model, skin=0.4)

    def call(hh):
        if next_call == "md":
            x = torch.empty_like(pos)
            nep.md_init(hh.h, pos, types, w.box, vel)
            nep.md_run(hh.h, 4, 1.0)
            nep.md_get_state(hh.h, pos=x)
            out = [x]
        elif next_call == "batch":
            out = list(hh.compute_batch(off, pos, types, boxes, per_atom=True).values())
        else:
            if next_call == "stats":
                nep.nep_get_stats(hh.h)
            out = list(hh.compute(pos, types, w.box, per_atom_virial=True).values())
        return [o.cpu().numpy() for o in out]

    expect = call(ref)
    for _ in range(2):
        nep.md_init(h.h, pos, types, w.box, vel)
        nep.nep_set_wait_limit(h.h, 1)
        nep.md_run_async(h.h, 3, 1.0)
        nep.nep_set_wait_limit(h.h, 0)
        for a, b in zip(call(h), expect):
            np.testing.assert_array_equal(a, b)
    ref.close()
    h.close()
