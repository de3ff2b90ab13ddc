"""The mixed student's two forms at the edges of the rule that chooses between them: one fused kernel, or (when a second
round of the fused kernel's resident blocks would be at most half full) a tensor-core descriptor kernel and a half-list
force kernel.  Either against the FP64 oracle on sampled atoms, within the mixed forms' bounds (operands of 8 or 11
significand bits: max 2e-2 / 3e-3 eV/Angstrom, RMSE 5 meV/Angstrom), and bitwise repeatable."""
import numpy as np
import pytest

import nep_inputs as ni
import oracle

pytestmark = pytest.mark.gpu

MAX_DF = {"mix_bf16": 2e-2, "mix_fp16": 3e-3}


@pytest.fixture(scope="module")
def api():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2604_24816_gb300 as pkg
    pkg.lib()
    return pkg


# multiples of half the resident atoms (five blocks of 128 on each SM), plus some atoms
@pytest.mark.parametrize("mode", ["mix_bf16", "mix_fp16"])
@pytest.mark.parametrize("halves, more, split", [(2, 0, False), (2, 1, True), (3, 0, True), (3, 1, False)])
def test_forms_at_the_rule_s_edges(api, student_params, student_model, mode, halves, more, split):
    import torch
    resident = 5 * 128 * torch.cuda.get_device_properties(0).multi_processor_count
    n = resident * halves // 2 + more
    nx = int(np.ceil((n / 4) ** (1 / 3)))
    wl = ni.fcc_cu_workload(0, sigma=0.05, seed=n % 1000, cells_xyz=(nx, nx, nx))
    pos = np.ascontiguousarray(wl.pos[:n])
    idx = np.random.default_rng(1).choice(n, 400, replace=False)
    Fo, Uo = oracle.forces_sampled(student_model, pos, wl.box, idx)
    with api.NEP(student_params, precision=mode) as nep:
        nep.set_state(pos, None, wl.box)
        nep.set_timing(True)
        E, F, W = nep.compute()
        assert (nep.timing()["descriptor"][1] > 0) == split
        nep.set_timing(False)
        U = nep.site_energies()
        E2, F2, W2 = nep.compute()
    d = F[idx] - Fo
    assert np.abs(d).max() <= MAX_DF[mode] and np.sqrt((d ** 2).mean()) <= 5e-3
    assert np.abs(U[idx] - Uo).max() <= MAX_DF[mode] / 10
    assert E2 == E and np.array_equal(F, F2) and np.array_equal(W, W2)
