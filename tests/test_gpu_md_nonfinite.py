"""Dynamics and relaxations whose positions leave the finite numbers end with NEP_ERR_NONFINITE,
whether a displacement overflows or is NaN from the start, and md_init makes the handle usable again."""
import numpy as np
import pytest

from paper_2205_10046_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("reps", [3, 26])  # 216 and 140,608 atoms: both forms of the rebuild
def test_nonfinite_positions_end_the_run(torch_cuda, reps):
    torch = torch_cuda
    from paper_2205_10046_gb300 import nep
    w = W.si_diamond(reps, seed=2)
    dev = lambda a, dt=torch.float64: torch.tensor(a, dtype=dt, device="cuda")  # noqa: E731
    pos, types, vel = dev(w.pos), dev(w.types, torch.int32), dev(w.vel)
    h = nep.NEP(w.model, skin=0.5)

    def good():
        nep.md_init(h.h, pos, types, w.box, vel)
        nep.md_run(h.h, 3, 1.0)
        x = torch.empty_like(pos)
        nep.md_get_state(h.h, pos=x)
        return x.cpu().numpy()

    ref = good()
    runs = {"run": lambda: nep.md_run(h.h, 3, 10.0), "ex": lambda: nep.md_run_ex(h.h, 3, 10.0, 1, dev(np.zeros((3, 4)))),
            "async": lambda: (nep.md_run_async(h.h, 3, 10.0), nep.md_status(h.h))}
    for bad in (1e308, float("nan")):  # 1e308 A/fs x 10 fs is infinite
        for run in runs.values():
            v = vel.clone()
            v[w.n_atoms // 2, 1] = bad
            nep.md_init(h.h, pos, types, w.box, v)
            with pytest.raises(nep.NepError) as e:
                run()
            assert e.value.code == -5
            with pytest.raises(nep.NepError) as e:
                nep.md_run(h.h, 1, 1.0)
            assert e.value.code == -7
    nep.md_init(h.h, pos, types, w.box)
    with pytest.raises(nep.NepError) as e:
        nep.fire_run(h.h, 5, 1e200, 0.0)
    assert e.value.code == -5
    np.testing.assert_array_equal(good(), ref)
    h.close()
