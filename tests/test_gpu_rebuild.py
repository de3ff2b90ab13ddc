"""The cell sort's forms at the sizes where they change: one block (up to 2,048 atoms and cells), one cluster (up to
16,384), a chain of kernels with several scan tiles, and more tiles than one pass of the carry scan holds.  The lists
must be those of a brute-force search, and the same rows again when the build starts from its own order."""
import numpy as np
import pytest

import nep_inputs as ni
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2604_24816_gb300 import build
    build.build()
    import paper_2604_24816_gb300 as pkg
    pkg.lib()
    return pkg


def _crystal(n, cells):
    pos, box = ni.student_cell(11 + n, cells, 0.05)
    return pos[:n], box


def _clusters(n, edge, seed):
    """Small fcc clusters scattered over a large empty box, some across its faces."""
    rng = np.random.default_rng(seed)
    pos, _ = ni.fcc_lattice(2, 2, 2)
    at = rng.uniform(0.0, edge, size=(-(-n // 32), 3))
    at[0] = 0.0                                     # on the corner: every axis wraps
    return (at[:, None, :] + pos[None] + rng.normal(0.0, 0.05, size=(len(at), 32, 3))).reshape(-1, 3)[:n], \
        np.array([edge, edge, edge])


CASES = {
    "1 atom": lambda: _crystal(1, (4, 4, 4)),
    "2047 atoms": lambda: _crystal(2047, (8, 8, 8)),
    "2048 atoms": lambda: _crystal(2048, (8, 8, 8)),
    "2049 atoms": lambda: _crystal(2049, (8, 8, 9)),
    "16384 atoms": lambda: _crystal(16384, (16, 16, 16)),
    "16385 atoms": lambda: _crystal(16385, (16, 16, 17)),
    "3000 atoms, 15625 cells": lambda: _clusters(3000, 150.5, 6),
    "3000 atoms, 17576 cells": lambda: _clusters(3000, 156.5, 7),
    "2016 atoms, 2197 cells": lambda: _clusters(2016, 80.0, 3),
    "1000 atoms, 4913 cells": lambda: _clusters(1000, 104.0, 4),
    "2500 atoms, 4.6M cells (1117 tiles)": lambda: _clusters(2500, 1000.0, 5),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_lists_are_those_of_a_brute_force_search(api, model_params, name):
    pos, box = CASES[name]()
    rl = model_params["rc_R"] + model_params["skin"]
    n = pos.shape[0]
    images = np.random.default_rng(n).integers(-2, 3, size=(n, 3)) * box       # unwrapped input
    with api.NEP(model_params) as nep:
        nep.set_state(pos + images, None, box)
        nep.build_neighbors()
        first = nep.neighbors(cap=160)
        nep.build_neighbors()                       # from the sorted order
        again = nep.neighbors(cap=160)
    for a, b in zip(first, again):
        assert np.array_equal(a, b)
    off, lst = oracle.neighbor_lists(np.mod(pos, box), box, rl, use_cells=False)
    counts, _, nown, rows = first
    assert nown.sum() * 2 == counts.sum()
    for i in range(n):
        differ = set(rows[i, :counts[i]].tolist()) ^ set(lst[off[i]:off[i + 1]].tolist())
        for j in differ:                            # only a pair within float32 rounding of the list radius may
            d = pos[j] - pos[i]
            d -= box * np.round(d / box)
            assert abs(np.linalg.norm(d) - rl) < 1e-5, (name, i, j)
