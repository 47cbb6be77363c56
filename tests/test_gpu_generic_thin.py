"""Run-time shapes with few angular sums: large calls take a thread per atom, smaller ones a warp. Both
forms on the same structures agree to FP32 rounding (relative 1e-5, the bar of either against the
oracle), alone, in batches, populations and dynamics, and the small ones meet the oracle."""
import numpy as np
import pytest

import oracle
from paper_2205_10046_gb300 import workloads as W

pytestmark = pytest.mark.gpu

THREADS = 49152  # atoms from which a thread per atom works; "wide" shapes: 131072

# n_max^R, N_bas^R, n_max^A, N_bas^A, N_neu, l_max^3b, 4b, 5b, types
SHAPES = {
    "smallest": (0, 0, 0, 0, 1, 1, 0, 0, 1),
    "four_body_on_l1": (3, 2, 3, 5, 7, 1, 2, 1, 3),
    "most_sums": (19, 19, 8, 19, 33, 2, 2, 1, 2),
    "most_n": (4, 7, 19, 3, 50, 1, 0, 1, 2),
    "l2_only": (8, 8, 1, 4, 40, 2, 0, 0, 2),
    "l3": (5, 4, 1, 4, 30, 3, 2, 1, 2),
    "l4": (6, 5, 0, 4, 20, 4, 2, 1, 3),
    "wide_l4": (4, 4, 2, 4, 20, 4, 2, 1, 2),
}


def _model(name, seed=7):
    nR, KR, nA, KA, H, l3, l4, l5, T = SHAPES[name]
    hyper = dict(n_types=T, rc_radial=4.5, rc_angular=3.5, n_max_radial=nR, n_max_angular=nA, basis_radial=KR,
                 basis_angular=KA, l_max_3b=l3, l_max_4b=l4, l_max_5b=l5, n_neuron=H)
    return W.random_model(hyper, seed, [W.MASS_C, W.MASS_SI, W.MASS_GE][:T])


def _close(a, b):
    assert np.linalg.norm(a - b) <= 1e-5 * max(np.linalg.norm(b), 1e-30)


@pytest.mark.parametrize("name", list(SHAPES))
def test_thread_and_warp_forms_agree(torch_cuda, name):
    torch = torch_cuda
    from paper_2205_10046_gb300 import nep
    model = _model(name)
    T = model.n_types
    threads = 131072 if name.startswith("wide") else THREADS
    parts = [W.random_structure(30 + n, n, n_types_model=T) for n in (33, 500, 127, 257)]
    few = W.concat_structures(parts)
    many = W.concat_structures(parts * (threads // few.n_atoms + 1))  # and an odd count of atoms
    assert few.n_atoms < threads <= many.n_atoms
    dev = lambda a, dt=torch.float64: torch.tensor(a, dtype=dt, device="cuda")  # noqa: E731
    h = nep.NEP(model, skin=0.4)
    batch = lambda b: {k: v.cpu().numpy() for k, v in h.compute_batch(  # noqa: E731
        b.offsets, dev(b.pos), dev(b.types, torch.int32), b.boxes, per_atom=True).items()}
    w, t = batch(few), batch(many)
    U, F, Wv = oracle.compute(model, *few.structure(0))
    _close(w["U"][:33], U)
    _close(w["F"][:33], F)
    for rep in (0, 1, many.n_struct // few.n_struct - 1):  # first, next and last copies
        a, s = rep * few.n_atoms, rep * few.n_struct
        for k in ("U", "F", "W"):
            _close(t[k][a:a + few.n_atoms], w[k])
        _close(t["E_struct"][s:s + few.n_struct], w["E_struct"])
        _close(t["W_struct"][s:s + few.n_struct], w["W_struct"])
    # one large structure: the sum of its atoms, its descriptors and a few steps
    pos, types, box = W.random_structure(3, threads + 5, n_types_model=T)
    p, ty = dev(pos), dev(types, torch.int32)
    o = {k: v.cpu().numpy() for k, v in h.compute(p, ty, box, per_atom_virial=True).items()}
    assert abs(o["E"][0] - o["U"].sum()) <= 1e-10 * np.abs(o["U"]).sum()
    q = dev(np.zeros((len(types), model.n_des)))
    nep.nep_descriptors(h.h, p, ty, box, q)
    sel = np.arange(0, len(types), 4099)
    Us, Fs, _ = oracle.compute(model, pos, types, box, sel=sel)
    _close(o["U"][sel], Us)
    _close(o["F"][sel], Fs)
    _close(q.cpu().numpy()[sel], oracle.descriptors(model, pos, types, box, sel=sel))
    nep.md_init(h.h, p, ty, box)
    rows = dev(np.zeros((3, 4)))
    nep.md_run(h.h, 3, 0.5, 1, rows)
    e = rows.cpu().numpy()[:, :2].sum(1)
    assert np.isfinite(e).all() and np.ptp(e) <= 1e-4 * len(types)
    h.close()


@pytest.mark.parametrize("name", ["smallest", "four_body_on_l1", "l2_only"])
def test_population_forms_agree(torch_cuda, name):
    """Losses of the same candidates in calls of few and of many members."""
    torch = torch_cuda
    from paper_2205_10046_gb300 import nep
    model = _model(name)
    b = W.concat_structures([W.random_structure(70 + k, 100 + k, n_types_model=model.n_types) for k in range(7)])
    dev = lambda a, dt=torch.float64: torch.tensor(a, dtype=dt, device="cuda")  # noqa: E731
    P = THREADS // b.n_atoms + 1
    z = dev(np.stack([_model(name, s).to_vector() for s in range(P)]))
    rng = np.random.default_rng(0)
    args = (b.offsets, dev(b.pos), dev(b.types, torch.int32), b.boxes, dev(rng.normal(size=b.n_struct)),
            dev(rng.normal(size=(b.n_atoms, 3))), dev(rng.normal(size=(b.n_struct, 6))), (1.0, 1.0, 1.0, 0.1, 0.1))
    h = nep.NEP(model, skin=0.4)
    many = nep.nep_eval_population(h.h, z, *args).cpu().numpy()
    few = nep.nep_eval_population(h.h, z[:3].contiguous(), *args).cpu().numpy()
    np.testing.assert_allclose(many[:3], few, rtol=1e-5)
    nep.nep_set_tuning(h.h, 5)  # members per launch do not change the form
    np.testing.assert_array_equal(nep.nep_eval_population(h.h, z, *args).cpu().numpy(), many)
    h.close()
