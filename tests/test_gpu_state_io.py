"""State and force transfers: pageable arrays of up to 4,096 atoms pass through page-locked staging that the kernels
read and write, larger ones through device copies; device and page-locked arrays are reached directly, positions and
velocities by one launch when both are and have the same alignment.  Every way moves the same doubles."""
import numpy as np
import pytest

import nep_inputs as ni

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2604_24816_gb300 as pkg
    pkg.lib()
    return pkg


def _arrays(kind, n):
    import torch
    if kind == "device":
        return torch.empty((n, 3), dtype=torch.float64, device="cuda")
    if kind == "device, 8 bytes off":
        return torch.empty(3 * n + 1, dtype=torch.float64, device="cuda")[1:].view(n, 3)
    if kind == "page-locked":
        return torch.empty((n, 3), dtype=torch.float64).pin_memory()
    return np.empty((n, 3))


def _host(a):
    return a if isinstance(a, np.ndarray) else a.cpu().numpy()


@pytest.mark.parametrize("n", [1, 255, 4096, 4097])
def test_every_way_moves_the_same_doubles(api, model_params, n):
    import torch
    pos, box = ni.student_cell(17, (11, 11, 10), 0.05, (0.0, 0.0, 0.0), 0)
    rng = np.random.default_rng(n)
    pos = pos[rng.permutation(pos.shape[0])[:n]] % box
    vel = 1e-3 * rng.standard_normal((n, 3))
    moved = pos + 0.01 * rng.standard_normal((n, 3))
    kinds = ["pageable", "device", "page-locked", "device, 8 bytes off"]
    want = None
    for kind in kinds:
        with api.NEP(model_params) as nep:
            for first, x in ((True, pos), (False, moved)):          # a new system, then an upload that keeps the list
                a, b = _arrays(kind, n), _arrays(kind, n)
                for dst, src in ((a, x), (b, vel)):
                    if isinstance(dst, np.ndarray):
                        dst[:] = src
                    else:
                        dst.copy_(torch.from_numpy(src))
                nep.set_state(a, b, box)
                E, F, W = nep.compute()
                t = nep.thermo()
            for kx, kv in ((kind, kind), (kind, "device"), ("pageable", "device, 8 bytes off")):
                ox, ov = _arrays(kx, n), _arrays(kv, n)
                nep.get_state(ox, ov)
                assert np.array_equal(_host(ov), vel)               # velocities come back as they went in
                d = _host(ox) - moved
                assert np.abs(d - box * np.round(d / box)).max() <= 8 * np.finfo(float).eps * box.max()
            got = (E, F, W, t["ke"])
        if want is None:
            want = got
        else:                                                       # fixed-point sums: bit for bit
            assert got[0] == want[0] and np.array_equal(got[1], want[1]) and np.array_equal(got[2], want[2])
            assert got[3] == want[3] > 0.0
