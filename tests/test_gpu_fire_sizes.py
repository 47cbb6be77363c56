"""FIRE velocity mixing by one cluster of thread blocks: sizes around the threads of a block and
of the cluster (128 x 8, 512 x 8), alone and as a served job, against the FP64 FIRE steps of the
oracle on forces of the same library.

Bar: positions within 1e-6 A after 8 steps of up to 1 fs. Forces of the same positions differ by
FP32 rounding, some 1e-6 eV/A, which moves an atom of 28 u by 1e-6 / (28 x 103.6) x 8^2 / 2, below
1e-7 A; the reductions are FP64 on both sides.
"""
import numpy as np
import pytest

import oracle
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


@pytest.mark.parametrize("n", [1, 127, 129, 1024, 1025, 4097])
def test_fire_sizes(torch_cuda, n):
    torch = torch_cuda
    from paper_2205_10046_gb300 import nep
    model = W.mixed_model(0)
    pos, types, box = W.random_structure(200 + n, n)
    t = torch.tensor(types, device="cuda")
    h = nep.NEP(model)

    def forces(x):
        g = h.compute(torch.tensor(x, device="cuda"), t, box)
        return g["E"].item(), g["F"].cpu().numpy()

    im = 1.0 / (np.asarray(model.mass)[types] * oracle.KAPPA)
    xo, _, _, steps_o, _ = oracle.fire_minimize(forces, pos, im, 8, 1.0, 1e-3)
    nep.md_init(h.h, torch.tensor(pos, device="cuda"), t, box)
    steps = nep.fire_run(h.h, 8, 1.0, 1e-3)
    p = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
    nep.md_get_state(h.h, pos=p)
    s = nep.Server(model, memory_budget=4 << 30, workers=2)
    jid = s.submit(nep.JOB_FIRE, pos, types, box, n_steps=8, dt_fs=1.0, fmax=1e-3)
    r = s.wait(60.0)
    ps = s.arrays(jid)[0]
    s.close()
    h.close()
    assert steps == steps_o and r["steps"] == steps_o
    for x in (p.cpu().numpy(), ps):
        f = (x - xo) @ np.linalg.inv(box)
        assert np.abs((f - np.round(f)) @ box).max() <= 1e-6
