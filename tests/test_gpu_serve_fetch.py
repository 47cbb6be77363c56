"""Results of served jobs that end together come over in bounded groups: more than one group's worth
at once, a job that is larger than a group by itself, and small ones after it."""
import numpy as np
import pytest

from paper_2205_10046_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_groups_of_results(torch_cuda):
    torch = torch_cuda
    from paper_2205_10046_gb300 import nep
    # 72 bytes an atom: 2,000,376 atoms take 137 MiB, 373,248 take 26
    sizes = [3, 36, 36, 63, 36, 36, 3, 36, 2]
    work = {r: W.si_diamond(r, seed=r, with_velocities=False) for r in set(sizes)}
    model = work[3].model
    h = nep.NEP(model, skin=0.4)
    ref = {}
    for r, w in work.items():
        out = h.compute(torch.tensor(w.pos, device="cuda"), torch.tensor(w.types, device="cuda"), w.box)
        ref[r] = out["E"].item(), out["F"].cpu().numpy()
    h.close()
    s = nep.Server(model, memory_budget=100 << 30, workers=64, skin=0.4)
    for _ in range(2):
        ids = [s.submit(nep.JOB_SINGLE, work[r].pos, work[r].types, work[r].box) for r in sizes]
        done = {}
        for _ in ids:
            res = s.wait(120.0)
            assert res is not None and res["status"] == 0, res
            done[res["id"]] = res
        for i, r in zip(ids, sizes):
            w, (E, F) = work[r], ref[r]
            pos, force, vel = s.arrays(i)
            # FP32 rounding of other pair orders; positions only wrapped
            assert abs(done[i]["energy"] - E) <= 1e-6 * w.n_atoms
            assert np.linalg.norm(force - F) <= 1e-5 * np.linalg.norm(F)
            f = (pos - w.pos) @ np.linalg.inv(w.box)
            assert np.abs((f - np.round(f)) @ w.box).max() <= 1e-9 and not vel.any()
    s.close()
