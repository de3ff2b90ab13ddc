"""The training kernels' groups of eight lanes at the edges of their ranges: cells of odd sizes (atoms past the last
one in a warp), batches that start inside the set, rows that do not start on a 16-byte boundary, and the parameter
gradient of a batch as the sum of its cells' gradients; and the fused loss against its plain form."""
import ctypes as C

import numpy as np
import pytest

import nep_inputs as ni

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env(trained_student_params):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2604_24816_gb300 import build
    build.build()
    from paper_2604_24816_gb300 import student as st
    rng = np.random.default_rng(3)
    cells = [ni.student_cell(40 + k, c, 0.07, (0.02, -0.01, 0.0), k + 1) for k, c in enumerate([(4, 4, 4), (4, 4, 5), (4, 5, 4)])]
    n = sum(p.shape[0] for p, _ in cells)
    cs = st.CellSet(cells, E=rng.normal(0.0, 1.0, 3), F=rng.normal(0.0, 0.1, (n, 3)))
    assert n % 4 != 0 and all(p.shape[0] % 2 for p, _ in cells[::2])
    qs = torch.tensor(np.asarray(trained_student_params["q_scale"], np.float32), device="cuda")
    return torch, st, cs, qs, st.pack(trained_student_params)


def _run(env, s0, s1, wE=1.0, wF=10.0, plain=False):
    torch, st, cs, qs, th = env
    theta = torch.tensor(th, device="cuda", requires_grad=True)
    E, F = st.student_ef(theta, qs, cs, s0, s1)
    loss = (st._loss_plain if plain else st.loss_fn)(E, F, cs, s0, s1, wE, wF)
    loss.backward()
    return E.detach(), F.detach(), loss.detach(), theta.grad


def test_batches_are_parts_of_the_set(env):
    torch, st, cs, qs, th = env
    E, F, _, _ = _run(env, 0, 3)
    for s0, s1 in ((0, 1), (1, 2), (1, 3), (2, 3)):
        e, f, _, _ = _run(env, s0, s1)
        a0, a1 = cs.atoms(s0, s1)
        assert torch.equal(e, E[s0:s1]) and torch.equal(f, F[a0:a1])


def test_gradient_is_the_sum_over_cells(env):
    """With a loss that is a sum over cells (each cell's mean weighted by its share)."""
    torch, st, cs, qs, th = env
    n = cs.n
    total = _run(env, 0, 3)[3].double()
    parts = torch.zeros_like(total)
    for s in range(3):
        a0, a1 = cs.atoms(s, s + 1)
        parts += _run(env, s, s + 1, 1.0 / 3.0, 10.0 * (a1 - a0) / n)[3].double()
    # float32 sums over some 1,000 atoms: errors add like their root at least, n at most, of 2^-24 of the terms
    assert (total - parts).abs().max() <= 1e-4 * total.abs().max()


def test_rows_off_a_16_byte_boundary(env):
    torch, st, cs, qs, th = env
    theta = torch.tensor(th, device="cuda")
    st.student_ef(theta, qs, cs)                       # fills cs.G
    rows = torch.zeros(cs.n * st.GS + 1, device="cuda")
    rows[1:] = cs.G.reshape(-1)
    F = [torch.zeros((cs.n, 3), device="cuda") for _ in range(2)]
    for out, ptr in zip(F, (cs.G.data_ptr(), rows.data_ptr() + 4)):
        rc = st.lib().st_force(0, cs.n, cs.n, cs.cap, st._p(cs.nbr), st._p(cs.dvec), st._p(cs.nnum), cs.rc, st._p(theta),
                               C.c_void_p(ptr), st._p(out), st._stream())
        assert rc == 0
    assert torch.equal(F[0], F[1]) and F[0].abs().max() > 0


@pytest.mark.parametrize("s0,s1", [(0, 3), (1, 2), (1, 3)])
def test_loss_matches_its_plain_form(env, s0, s1):
    torch, st, cs, qs, th = env
    fused, plain = _run(env, s0, s1), _run(env, s0, s1, plain=True)
    assert abs(float(fused[2] - plain[2])) <= 1e-13 * abs(float(plain[2]))    # float64 sums in another order
    assert (fused[3] - plain[3]).abs().max() <= 1e-6 * plain[3].abs().max()   # one float32 rounding of each dL/dF


def test_loss_keeps_what_autograd_could_do(env):
    """A second derivative, other strides, and a call under forward mode give what the plain form gives."""
    torch, st, cs, qs, th = env
    a0, a1 = cs.atoms(1, 3)
    g = torch.Generator(device="cuda").manual_seed(1)
    E = torch.randn(2, generator=g, device="cuda", dtype=torch.float64, requires_grad=True)
    F = torch.randn((a1 - a0, 3), generator=g, device="cuda", requires_grad=True)

    def second(loss):
        gE, gF = torch.autograd.grad(loss(E, F, cs, 1, 3), (E, F), create_graph=True)
        return torch.autograd.grad((gE * gE).sum() + (gF * gF).sum().double(), (E, F))

    for a, b in zip(second(st.loss_fn), second(st._loss_plain)):
        assert torch.allclose(a, b, rtol=1e-5)
    strided = F.detach().t().contiguous().t()
    assert torch.allclose(st.loss_fn(E, strided, cs, 1, 3), st._loss_plain(E, strided, cs, 1, 3), rtol=1e-12)
    import torch.autograd.forward_ad as fwad
    with fwad.dual_level():
        dual = fwad.make_dual(F.detach(), torch.ones_like(F))
        t = [fwad.unpack_dual(f(E.detach(), dual, cs, 1, 3)).tangent for f in (st.loss_fn, st._loss_plain)]
    assert torch.allclose(t[0], t[1], rtol=1e-6)


def test_loss_gradient_is_of_the_value_returned(env):
    """Labels, energies and forces replaced or rewritten between the loss and its backward pass: the gradient stays that
    of the loss returned, once and as a second derivative."""
    torch, st, cs, qs, th = env
    a0, a1 = cs.atoms(1, 3)
    g = torch.Generator(device="cuda").manual_seed(2)
    E0 = torch.randn(2, generator=g, device="cuda", dtype=torch.float64)
    F0 = torch.randn((a1 - a0, 3), generator=g, device="cuda")
    keep = cs.E_ref, cs.F_ref

    def swap(E, F):
        cs.E_ref, cs.F_ref = keep[0] + 1.0, keep[1] - 2.0

    def rewrite(E, F):
        cs.E_ref.mul_(3.0)
        cs.F_ref.zero_()

    def outputs(E, F):
        with torch.no_grad():
            E.zero_()
            F.mul_(-1.0)

    def derivatives(loss, change):
        cs.E_ref, cs.F_ref = keep[0].clone(), keep[1].clone()
        x, y = E0.clone().requires_grad_(), F0.clone().requires_grad_()
        E, F = x * 1.0, y * 1.0
        value = loss(E, F, cs, 1, 3)
        change(E, F)
        first = torch.autograd.grad(value, (x, y), retain_graph=True)
        gE, gF = torch.autograd.grad(value, (x, y), create_graph=True)
        return (*first, *torch.autograd.grad((gE * gE).sum() + (gF * gF).sum().double(), (x, y)))

    try:
        for change in (swap, rewrite, outputs):
            for a, b in zip(derivatives(st.loss_fn, change), derivatives(st._loss_plain, change)):
                assert b.abs().max() > 0 and torch.allclose(a, b, rtol=1e-5), change.__name__
    finally:
        cs.E_ref, cs.F_ref = keep
    # and through hooks on what is saved
    with torch.autograd.graph.save_on_cpu():
        a, b = _run(env, 0, 3)[3], _run(env, 0, 3, plain=True)[3]
    assert (a - b).abs().max() <= 1e-6 * b.abs().max()


def test_gradient_of_many_atoms_is_summed_in_float64(env):
    """Equal atoms without directional derivatives, so that every term of a parameter has one sign (c_A's, which come from
    eight components of two degrees, left out): a lane adds at most 32 atoms' two products in float32 and the block 2 + 8
    partial sums, each with a relative error of 2^-24 or less; the product itself and the result are rounded once more."""
    torch, st, cs, qs, th = env
    n = 12_000_000
    theta = torch.tensor(th, device="cuda")
    full = lambda *shape: torch.ones(shape, device="cuda")
    Q, S, zero = full(n, st.KB) * cs.Q[:1], full(n, st.NSB) * cs.S[:1], torch.zeros(n * st.NSB, device="cuda")
    pos = torch.zeros((n, 4), device="cuda")                       # cell 0
    gE = torch.tensor([0.7], dtype=torch.float64, device="cuda")

    def grad(m):
        out = torch.empty(st.NPAR, device="cuda")
        ws = torch.empty(int(st.lib().st_grad_scratch(0, m)), device="cuda")
        rc = st.lib().st_grad(0, m, st._p(theta), st._p(qs), st._p(pos), st._p(Q), st._p(S), st._p(zero), st._p(zero),
                              st._p(gE), st._p(ws), st._p(out), st._stream())
        assert rc == 0
        return out.double()

    one, many = grad(1) * n, grad(n)
    for o, m in ((0, 32), (64, st.NPAR - 64)):                     # c_R; W0, b0, w1, b1
        a, b = one[o:o + m], many[o:o + m]
        assert a.abs().min() > 0 and ((a - b).abs() / a.abs()).max() <= 76 * 2.0 ** -24
