"""The wide kernels (several lanes per atom) at the atom counts where the number of lanes changes, one more than a
full warp or block of them, a single atom without neighbours, and each form of the network; and the fallback
model's list on both sides of the count where its split changes.  Against the FP64 oracle, with the bounds of the
one-thread-per-atom kernels' tests."""
import numpy as np
import pytest

import nep_inputs as ni
import oracle

pytestmark = pytest.mark.gpu

# lanes per atom: 32 up to 1,024 atoms, 16 up to 4,096, 8 up to 9,728, 4 up to 19,456, then one thread per atom
SIZES = [1, 5, 129, 1024, 1025, 4096, 4097, 9728, 9729, 19456, 19457]


@pytest.fixture(scope="module")
def api():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2604_24816_gb300 import build
    build.build()
    import paper_2604_24816_gb300 as pkg
    pkg.lib()
    return pkg


def _cell(n):
    """n atoms of a displaced crystal: the last ones missing from the box, so rows differ in length."""
    c = max(4, int(np.ceil((n / 4) ** (1 / 3))))
    pos, box = ni.student_cell(700 + n, (c, c, c + (4 * c ** 3 < n)), 0.05, (0.01, 0.0, -0.01))
    return pos[:n], box


@pytest.mark.parametrize("n", SIZES)
def test_teacher(api, model_params, model, n):
    pos, box = _cell(n)
    Eo, Uo, Fo, Wo = oracle.energy_forces(model, pos, box)
    with api.NEP(model_params) as nep:
        nep.set_state(pos, None, box)
        E, F, W = nep.compute()
        U, q = nep.site_energies(), nep.descriptors()
        again = nep.compute()
    qo = oracle.descriptors(model, pos, box)
    assert np.array_equal(F, again[1]) and E == again[0] and np.array_equal(W, again[2])
    assert np.abs(F - Fo).max() <= 1e-4
    assert abs(E - Eo) <= 1e-6 * abs(Eo) + 1e-6
    assert np.abs(U - Uo).max() <= 1e-5
    assert np.abs(W - Wo).max() <= 1e-5 * max(np.abs(Wo).max(), 1.0)
    assert (np.abs(q - qo).max(0) <= 2e-5 * np.maximum(np.abs(qo).max(0), 1.0)).all()


@pytest.mark.parametrize("precision", ["mix_bf16", "mix_fp16"])
@pytest.mark.parametrize("n", [5, 1024, 1025, 4097, 9729, 19457])
def test_mixed(api, model_params, model, trained_student_params, n, precision):
    # the bounds of the tensor-core forms' tests: RMSE 5 meV/A, largest 20 (bf16) or 3 meV/A (f16)
    pos, box = _cell(n)
    for params, om in ((model_params, model), (trained_student_params, oracle.Model(trained_student_params))):
        Fo = oracle.energy_forces(om, pos, box)[2]
        with api.NEP(params, precision=precision) as nep:
            nep.set_state(pos, None, box)
            dF = nep.compute()[1] - Fo
        assert np.sqrt(np.mean(dF ** 2)) <= 5e-3
        assert np.abs(dF).max() <= (2e-2 if precision == "mix_bf16" else 3e-3)


@pytest.mark.parametrize("n", [1, 1024, 1025, 4097, 9729, 19457])
def test_student(api, trained_student_params, n):
    pos, box = _cell(n)
    Eo, Uo, Fo, Wo = oracle.energy_forces(oracle.Model(trained_student_params), pos, box)
    with api.NEP(trained_student_params) as nep:
        nep.set_state(pos, None, box)
        E, F, W = nep.compute()
    assert np.abs(F - Fo).max() <= 1e-4
    assert abs(E - Eo) <= 1e-6 * abs(Eo) + 1e-6
    assert np.abs(W - Wo).max() <= 1e-5 * max(np.abs(Wo).max(), 1.0)


@pytest.mark.parametrize("n,share", [(257, 0.5), (1024, 1.0), (4096, 1.0), (4097, 1.0), (20000, 0.03), (20000, 0.4)])
def test_fallback_list(api, model_params, model, trained_student_params, n, share):
    """1 to 4,096 flagged atoms take a warp each, more a quarter of one; the student's own kernel is a wide one
    up to 19,456 atoms."""
    pos, box = _cell(n)
    sm = oracle.Model(trained_student_params)
    qt = oracle.descriptors(sm, pos, box) * np.asarray(trained_student_params["q_scale"], np.float32)
    lo, hi = qt.min(0) - 1.0, qt.max(0) + 1.0
    if share < 1.0:
        hi[0] = np.sort(qt[:, 0])[int(n * (1 - share)) - 1]
        gap = np.sort(np.abs(qt[:, 0] - hi[0]))[1]     # the threshold between two atoms' descriptors
        hi[0] += 0.5 * gap
    else:
        hi[0], lo[0] = lo[0] - 1.0, lo[0] - 2.0
    with api.NEP(trained_student_params) as nep:
        nep.set_fallback(model_params, lo, hi, margin=0.0, max_fraction=1.0)
        nep.set_state(pos, None, box)
        E, F, W = nep.compute()
        flags, count = nep.fallback()
    assert count == flags.sum() and abs(count - share * n) <= 2
    Eo, Uo, Fo, Wo = oracle.energy_forces_select(sm, model, flags, pos, box)
    assert np.abs(F - Fo).max() <= 1e-4
    assert abs(E - Eo) <= 1e-6 * abs(Eo)
    assert np.abs(W - Wo).max() <= 1e-5 * np.abs(Wo).max()
