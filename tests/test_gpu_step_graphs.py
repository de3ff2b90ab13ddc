"""MD steps from replayed graphs above the sizes whose cell sort is one kernel: every step's rebuild chain sits behind a
conditional node, one step per graph at first and several when enough steps have been asked for.  Any grouping of the steps
into calls gives the bits, rebuilds, evaluations and flagged atoms of single steps and of launches one by one."""
import numpy as np
import pytest

import nep_inputs as ni

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


# (dt, steps) of the calls: one step per graph until 80 steps have been asked for, then ten (8 times their own length),
# with a remainder and a call too short for them; another dt, and a call long enough to get its graph of 16 at once; back
CALLS = [(1.0, 10)] * 10 + [(1.0, 25), (1.0, 3), (0.5, 7), (0.5, 150), (1.0, 5)]
SINGLE = [(dt, 1) for dt, k in CALLS for _ in range(k)]
# lanes per atom and a cell sort in a chain of kernels; the fused kernels; the two-kernel form
CASES = {
    "teacher 17408": ("teacher", "fp32", (16, 16, 17)),
    "teacher 22032": ("teacher", "fp32", (18, 18, 17)),
    "student with fallback 22032": ("student", "fp32", (18, 18, 17)),
    "student with fallback, bf16, 108000": ("student", "mix_bf16", (30, 30, 30)),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_grouping_with_conditional_chains(api, model_params, trained_student_params, name):
    kind, precision, cells = CASES[name]
    sp = trained_student_params
    wl = ni.fcc_cu_workload(0, temperature=600.0, sigma=0.06, seed=5, cells_xyz=cells)

    def run(calls, timing=False):
        with api.NEP(model_params if kind == "teacher" else sp, rebuild_every=4, precision=precision) as nep:
            nep.set_state(wl.pos, wl.vel, wl.box)
            if kind == "student":                    # a limit of the first descriptor that some atoms are beyond
                q = nep.descriptors()[:, 0] * np.float32(sp["q_scale"][0])
                lo, hi = np.full(12, -1e3), np.full(12, 1e3)
                hi[0] = np.percentile(q, 95)
                nep.set_fallback(model_params, lo, hi, margin=0.0, max_fraction=1.0)
            nep.compute(forces=False)
            nep.set_timing(timing)
            c0 = nep.counters()
            for dt, k in calls:
                nep.step(dt, k)
            flags = nep.fallback() if kind == "student" else (None, 0)
            c1 = nep.counters()
            return (*nep.get_state(), flags[0]), nep.thermo(), {k: c1[k] - c0[k] for k in c1}

    arrays, thermo, count = run(CALLS)
    steps = sum(k for _, k in CALLS)
    assert count["steps"] == count["evaluations"] == steps and count["rebuilds"] >= steps // 4
    if kind == "student":
        assert 0 < arrays[2].sum() < wl.n and count["fallback_atoms"] > 0
    for calls, timing in ((SINGLE, False), (CALLS, True)):
        other, th, c = run(calls, timing)
        for a, b in zip(arrays, other):
            assert a is None or np.array_equal(a, b)
        for k in thermo:
            assert np.array_equal(thermo[k], th[k]), k
        launches, more = count.pop("launches"), c.pop("launches")
        assert count == c
        count["launches"] = launches
        if not timing:                               # the closing kick of every call; the chains run on rebuild steps only
            assert more - launches == len(SINGLE) - len(CALLS)


def test_a_long_call_after_a_short_one(api, model_params):
    """Small systems: the graph of a short first call, and the one that replaces it in a call of 256 steps."""
    wl = ni.fcc_cu_workload(4, 300.0, 0.05, seed=6)

    def run(calls):
        with api.NEP(model_params, rebuild_every=7) as nep:
            nep.set_state(wl.pos, wl.vel, wl.box)
            for k in calls:
                nep.step(1.0, k)
            return (*nep.get_state(), nep.thermo()["pe"], nep.counters()["rebuilds"])

    for a, b in zip(run([4, 20, 260, 5]), run([1] * 289)):
        assert np.array_equal(a, b)
