"""The autotuner keeps the default block size where the kernels of a small set read none (a choice
between equal launches is noise), and its population times stand for nep_eval_population's kernels."""
import numpy as np
import pytest

from paper_2205_10046_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _set(torch, n_struct):
    b = W.batch_structures(n_struct, seed=8)
    return b, torch.tensor(b.pos, device="cuda"), torch.tensor(b.types, dtype=torch.int32, device="cuda")


def test_small_sets_keep_the_default(torch_cuda):
    from paper_2205_10046_gb300 import nep
    b, p, t = _set(torch_cuda, 32)
    assert b.n_atoms <= 14592
    h = nep.NEP(W.mixed_model(0))
    for _ in range(4):
        nep.nep_set_tuning(h.h, 0, 0, 0, 1)
        tune = nep.nep_autotune(h.h, b.offsets, p, t, b.boxes, 0)
        assert (tune["atom_block"], tune["gather_block"]) == (128, 128)
        assert tune["best_ms"] == tune["default_ms"]
    h.close()


@pytest.mark.parametrize("n_pop", [1, 3, 8])
def test_population_sets(torch_cuda, n_pop):
    torch = torch_cuda
    from paper_2205_10046_gb300 import nep
    b, p, t = _set(torch, 24)
    model = W.mixed_model(0)
    h = nep.NEP(model)
    z = torch.tensor(np.stack([W.mixed_model(k).to_vector() for k in range(n_pop)]), device="cuda")
    e, f = torch.zeros(b.n_struct, dtype=torch.float64, device="cuda"), torch.zeros_like(p)
    base = nep.nep_eval_population(h.h, z, b.offsets, p, t, b.boxes, e, f).cpu().numpy()
    nep.nep_set_tuning(h.h, 0, 0, 0, 1)
    tune = nep.nep_autotune(h.h, b.offsets, p, t, b.boxes, n_pop)
    sizes = [m for m in (1, 2, 4, 8) if m <= n_pop]
    # six pairs of block sizes, one member with the defaults, the members per launch
    assert tune["n_tried"] == 6 + (n_pop > 1) + len(sizes) and tune["members_per_launch"] in sizes
    if n_pop == 1:  # the per-atom kernel of one member on a small set takes no block size
        assert tune["atom_block"] == 128
    assert 0 < tune["best_ms"] and 0 < tune["default_ms"]
    got = nep.nep_eval_population(h.h, z, b.offsets, p, t, b.boxes, e, f).cpu().numpy()
    np.testing.assert_allclose(got, base, rtol=1e-12, atol=1e-15)  # the order of the force error's sums
    h.close()
