"""Ranges of cells that student_ef accepts, and which calls of the training loss reach the fused kernels, which read the labels by address: on the CPU,
with host tensors that report themselves as CUDA ones.  Every other call takes the loss in PyTorch operations."""
from types import SimpleNamespace

import numpy as np
import pytest
import torch

from paper_2604_24816_gb300 import student as st

SIZES = (3, 5, 4)


def _cells(**other):
    start = np.concatenate([[0], np.cumsum(SIZES)]).astype(np.int64)
    c = SimpleNamespace(n_cells=3, n=12, start_h=start, E_ref=torch.randn(3, dtype=torch.float64), F_ref=torch.randn(12, 3),
                        natoms=torch.tensor(SIZES, dtype=torch.float64))
    c.atoms = lambda s0, s1: (int(start[s0]), int(start[s1]))
    for k, v in other.items():
        setattr(c, k, v)
    return c


@pytest.fixture(autouse=True)
def cuda_tensors(monkeypatch):
    monkeypatch.setattr(torch.Tensor, "is_cuda", property(lambda self: True))


def _outputs(c, s0, s1):
    a0, a1 = c.atoms(s0, s1)
    return torch.randn(s1 - s0, dtype=torch.float64), torch.randn(a1 - a0, 3)


def _fused(c, s0=0, s1=3, outputs=None):
    return st._takes_fused_loss(*(outputs or _outputs(c, s0, s1)), c, s0, s1, 1.0, 10.0)


def test_labels_of_the_set_take_the_kernels():
    assert _fused(_cells()) and _fused(_cells(), 1, 3) and _fused(_cells(), 2, 3)


SHORT = {
    "energies": dict(E_ref=torch.zeros(2, dtype=torch.float64)),
    "forces": dict(F_ref=torch.zeros(11, 3)),
    "no energies": dict(E_ref=torch.zeros(0, dtype=torch.float64)),
}


@pytest.mark.parametrize("name", sorted(SHORT))
def test_labels_too_few_are_refused(name):
    c = _cells(**SHORT[name])
    out = _outputs(c, 0, 3)
    assert not _fused(c, outputs=out)
    with pytest.raises(RuntimeError):               # sizes that do not match
        st.loss_fn(*out, c, 0, 3)


OTHER = {
    "one energy for every cell": dict(E_ref=torch.tensor([0.25], dtype=torch.float64)),
    "energies as a column": dict(E_ref=torch.randn(3, 1, dtype=torch.float64)),
    "one force for every atom": dict(F_ref=torch.randn(1, 3)),
    "more energies than cells": dict(E_ref=torch.randn(7, dtype=torch.float64)),
    "another type of atom counts": dict(natoms=torch.tensor(SIZES, dtype=torch.float32)),
    "differentiated energies": dict(E_ref=torch.randn(3, dtype=torch.float64, requires_grad=True)),
}


@pytest.mark.parametrize("name", sorted(OTHER))
def test_other_labels_take_the_plain_loss(name):
    c = _cells(**OTHER[name])
    out = _outputs(c, 0, 3)
    assert not _fused(c, outputs=out)
    assert torch.equal(st.loss_fn(*out, c, 0, 3), st._loss_plain(*out, c, 0, 3))


def test_labels_on_another_device_do_not_reach_the_kernels():
    for k in ("E_ref", "F_ref", "natoms"):
        c = _cells()
        setattr(c, k, getattr(c, k).to("meta"))
        assert not _fused(c)


def test_a_set_without_labels_raises_as_the_plain_loss_does():
    for k in ("E_ref", "F_ref"):
        with pytest.raises(TypeError):
            c = _cells(**{k: None})
            st.loss_fn(*_outputs(c, 0, 3), c, 0, 3)


def test_ranges_from_the_end_take_the_plain_loss():
    c = _cells()
    out = torch.randn(1, dtype=torch.float64), torch.randn(5, 3)
    assert not _fused(c, -3, -2, outputs=out)
    assert torch.equal(st.loss_fn(*out, c, -3, -2), st._loss_plain(*out, c, -3, -2))


class _Calls:
    """Records the kernel library's calls (every one succeeds)."""

    def __init__(self):
        self.args = {}

    def __getattr__(self, name):
        return lambda *a: self.args.setdefault(name, a) and 0


@pytest.fixture
def calls(monkeypatch):
    L = _Calls()
    monkeypatch.setattr(st, "lib", lambda: L)
    monkeypatch.setattr(st, "_stream", lambda: None)
    return L


def _resident(c):
    for k, shape in dict(pos=(12, 4), Q=(12, 8), S=(12, 64), U=(12,), G=(12, 40), nbr=(96, 12), dvec=(96, 12, 4), nnum=(12,),
                         dQ=(12, 8), dS=(12, 64), scratch=(289,), start=(4,)).items():
        setattr(c, k, torch.zeros(shape))
    c.cap, c.rc = 96, st.st_cutoffs(5.0, 4.0)
    return c


@pytest.mark.parametrize("as_int", [int, np.int64, np.int32, torch.tensor])
def test_ranges_of_any_integer_type(calls, as_int):
    c = _resident(_cells())
    theta, qs = torch.zeros(st.NPAR, requires_grad=True), torch.ones(12)
    E, F = st.student_ef(theta, qs, c, as_int(1), as_int(3))
    assert E.shape == (2,) and F.shape == (9, 3)
    assert calls.args["st_energy"][-2].value == E.data_ptr() - 8 and calls.args["st_force"][-2].value == F.data_ptr() - 36
    (E.sum() + F.sum().double()).backward()
    assert theta.grad.shape == (st.NPAR,)


def test_an_empty_range(calls):
    c = _resident(_cells())
    theta = torch.zeros(st.NPAR, requires_grad=True)
    for s0, s1 in ((1, 1), (2, 1)):
        E, F = st.student_ef(theta, torch.ones(12), c, s0, s1)
        assert E.shape == (0,) and F.shape == (0, 3)
        (E.sum() + F.sum().double()).backward()


def test_a_fraction_is_no_cell(calls):
    c = _resident(_cells())
    with pytest.raises((TypeError, IndexError)):
        st.student_ef(torch.zeros(st.NPAR), torch.ones(12), c, 0.5, 3)
