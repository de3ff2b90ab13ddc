"""The work that programs built on this framework have it do, as cases that can be timed and compared.

    listed()            the cases; draw(rng) gives another one of the same ranges
    prepare(case, seed) inputs and the handles or plans a program keeps, on the GPU
    run(state)          one pass through the public entry points, returning what they compute
    work(case)          bytes and float32 operations a pass cannot do without
    tolerance(case)     how far another correct implementation at the same precision may be off
    exact(case, seed)   the outputs in 64 bits, in plain torch

Paths ("path" of a case):
    md         a block of velocity-Verlet steps of a resident system, then its state and thermodynamics
    label      energies, forces and virials of the snapshots of one small cell, uploaded from the host
    train      one optimiser step of the student: forward, loss, backward, Adam
    eval       the student's energies and forces over a whole held-out set
    noalloc    one force evaluation through the allocation-free C entry point
    roundtrip  upload from page-locked memory, one step, download: a host program that owns the state
"""
from __future__ import annotations

import ctypes as C
import json
import math
import os

import numpy as np
import torch

from paper_2604_24816_gb300 import NEP, load_model
from paper_2604_24816_gb300 import nep as _nep
from paper_2604_24816_gb300 import student as _st

_PARAMS = os.path.join(os.path.dirname(os.path.abspath(_nep.__file__)), "params")
_TEACHER = os.path.join(_PARAMS, "cu_nep4_synth.json")
_STUDENT = os.path.join(_PARAMS, "cu_student_trained.json")
A_CU = 3.615                       # fcc lattice constant (Angstrom)
KB = 8.617333262e-5                # eV/K
KE = 103.642696562                 # 1 amu Angstrom^2/fs^2 in eV
ACC = 9.64853321233100e-3          # (eV/Angstrom)/amu in Angstrom/fs^2
FORMS = ("plain", "mix_bf16", "mix_fp16", "student", "student_fb", "student_bf16_fb")
E0 = -0.046                        # mean site energy of the trained student (eV): where synthetic labels are centred


def _md(name, form, nx, ny, nz, T, steps=10, strain=0.0, vac=0, void=0.0):
    return dict(name=name, path="md", form=form, nx=nx, ny=ny, nz=nz, T=T, steps=steps, strain=strain, vac=vac,
                void=void)


def listed():
    return [
        # the smallest system a periodic cell allows: equilibration and short trajectories, all latency
        _md("md_plain_256", "plain", 4, 4, 4, 300.0),
        # a small mixed-precision system, ragged: not a multiple of a block, strained, with vacancies
        _md("md_mix_fp16_1k", "mix_fp16", 6, 7, 6, 700.0, strain=0.015, vac=3),
        # a mid-size teacher run (the CPU baseline's cell): a fraction of one wave of blocks
        _md("md_plain_16k", "plain", 16, 16, 16, 300.0),
        # the student as deployed, in float32
        _md("md_student_56k", "student", 24, 23, 26, 600.0),
        # the student with the teacher as per-atom fallback on a strained void, bf16 network
        _md("md_student_fb_void", "student_bf16_fb", 32, 32, 32, 300.0, strain=0.02, void=20.0),
        # the headline system
        _md("md_plain_1M", "plain", 64, 64, 64, 300.0),
        # a large hot system in mixed precision
        _md("md_mix_bf16_8M", "mix_bf16", 128, 128, 128, 1200.0),
        # labels for training: one trajectory's snapshots of a small strained cell with vacancies, no pair term
        dict(name="label_862", path="label", nx=6, ny=6, nz=6, T=900.0, strain=-0.02, vac=2, snapshots=8),
        # a training step on the distillation's mini-batch of 40 mixed cells
        dict(name="train_40", path="train", cells=40, T=900.0),
        # the student over a held-out set
        dict(name="eval_200", path="eval", cells=200, T=900.0),
        # a plugin's force call
        dict(name="noalloc_4k", path="noalloc", nx=10, ny=10, nz=10, T=300.0, strain=0.0, vac=0),
        # a host program that owns the state and steps it one at a time
        dict(name="roundtrip_262k", path="roundtrip", form="plain", nx=40, ny=40, nz=41, T=300.0, strain=0.0, vac=0,
             void=0.0),
    ]


def _cells(rng, lo, hi):
    """Conventional cells per edge, their product spread over the logarithm of [lo, hi], edges unequal."""
    c = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    e = [max(4, round(c ** (1 / 3) * rng.uniform(0.85, 1.18))) for _ in range(2)]
    return e[0], e[1], max(4, min(round(c / (e[0] * e[1])), hi // (e[0] * e[1])))


def draw(rng):
    path = rng.choice(["md", "md", "md", "label", "train", "eval", "noalloc", "roundtrip"])
    T, strain = round(rng.uniform(300.0, 1200.0), 1), round(rng.uniform(-0.02, 0.02), 4)
    if path in ("md", "roundtrip"):
        form = rng.choice(FORMS)
        nx, ny, nz = _cells(rng, 64, 64 ** 3 if path == "md" else 40 ** 3)
        # a fallback form is for what leaves the training range: about half of them hold a void
        void = round(0.22 * A_CU * min(nx, ny, nz), 2) if "fb" in form and min(nx, ny, nz) >= 8 and rng.random() < 0.5 else 0.0
        c = dict(path=path, form=form, nx=nx, ny=ny, nz=nz, T=T, strain=strain, vac=rng.randrange(0, 1 + nx * ny * nz // 50),
                 void=void)
        if path == "md":
            c["steps"] = rng.choice([1, 3, 10, 25]) if nx * ny * nz < 30000 else 10
        return c
    if path == "label":
        nx, ny, nz = (rng.randint(4, 6) for _ in range(3))
        return dict(path=path, nx=nx, ny=ny, nz=nz, T=T, strain=strain, vac=rng.randint(1, 4), snapshots=rng.randint(2, 12))
    if path == "train":
        return dict(path=path, cells=round(math.exp(rng.uniform(math.log(4), math.log(160)))), T=T)
    if path == "eval":
        return dict(path=path, cells=round(math.exp(rng.uniform(math.log(20), math.log(400)))), T=T)
    nx, ny, nz = _cells(rng, 64, 2000)
    return dict(path=path, nx=nx, ny=ny, nz=nz, T=T, strain=strain, vac=rng.randint(0, 5))


# ---------------------------------------------------------------------------------------------------
# inputs

def _crystal(case, gen, dev):
    """Positions of a strained fcc crystal with vacancies or a void, thermally displaced, and its box.  The
    lattice is shifted by a quarter of its constant, so that no atom sits on the periodic boundary."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    ix = torch.arange(nx * ny * nz, device=dev)
    cell = torch.stack([ix // (ny * nz), ix // nz % ny, ix % nz], 1).double()
    basis = torch.tensor([[0.0, 0.0, 0.0], [0.5, 0.5, 0.0], [0.5, 0.0, 0.5], [0.0, 0.5, 0.5]], device=dev).double()
    pos = ((cell[:, None, :] + basis[None]) + 0.25).reshape(-1, 3) * A_CU
    box = np.array([nx, ny, nz], dtype=np.float64) * A_CU
    if case.get("void"):
        mid = torch.tensor(box / 2, device=dev)
        pos = pos[((pos - mid) ** 2).sum(1) >= case["void"] ** 2]
    if case.get("vac"):
        pos = pos[torch.randperm(pos.shape[0], generator=gen, device=dev)[case["vac"]:].sort().values]
    scale = np.array([1.0, 1.0, 1.0 + case["strain"]])
    box = box * scale
    pos = pos * torch.tensor(scale, device=dev)
    pos = pos + 0.05 * math.sqrt(case["T"] / 300.0) * torch.randn(pos.shape, generator=gen, device=dev,
                                                                 dtype=torch.float64)
    return torch.remainder(pos, torch.tensor(box, device=dev)), box


def _velocities(n, T, mass, gen, dev):
    v = torch.randn((n, 3), generator=gen, device=dev, dtype=torch.float64) * math.sqrt(KB * T / mass / KE)
    return v - v.mean(0)


def _gen(seed, dev):
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    return g


def _model(path):
    with open(path) as f:
        return json.load(f)


# fcc cells of 256 to 864 atoms, as the distillation's trajectories use
_TRAIN_SIZES = [(4, 4, 4), (4, 4, 5), (4, 5, 5), (5, 5, 5), (4, 5, 6), (5, 5, 6), (5, 6, 6), (6, 6, 6)]


def _train_inputs(case, seed, dev):
    """Cells (positions, box) of mixed sizes, strains and vacancies, with labels around the student's energies
    and thermal force magnitudes."""
    gen = _gen(seed, dev)
    r, sizes = np.random.default_rng(seed), np.random.default_rng(case["cells"])
    cells, E, F = [], [], []
    for _ in range(case["cells"]):
        nx, ny, nz = _TRAIN_SIZES[int(sizes.integers(len(_TRAIN_SIZES)))]
        c = dict(nx=nx, ny=ny, nz=nz, T=case["T"], strain=float(r.uniform(-0.03, 0.03)), vac=int(sizes.integers(1, 5)))
        pos, box = _crystal(c, gen, dev)
        cells.append((pos.cpu().numpy(), box))
        E.append(pos.shape[0] * (E0 + 0.002 * float(r.standard_normal())))
        F.append(0.06 * r.standard_normal((pos.shape[0], 3)))
    return cells, np.array(E), np.concatenate(F).astype(np.float32)


class _Run:
    """What a program holds between calls."""


def prepare(case, seed):
    dev = torch.device("cuda")
    s = _Run()
    s.path, s.case = case["path"], case
    if s.path in ("train", "eval"):
        cells, E, F = _train_inputs(case, seed, dev)
        m = _model(_STUDENT)
        s.cells = _st.CellSet(cells, E=E, F=F)
        s.qs = torch.tensor(np.asarray(m["q_scale"], np.float32), device=dev)
        s.theta = torch.tensor(_st.pack(m), device=dev, requires_grad=s.path == "train")
        if s.path == "train":
            s.m, s.v, s.t = torch.zeros_like(s.theta), torch.zeros_like(s.theta), 0
        return s
    gen = _gen(seed, dev)
    if s.path == "label":
        x, s.box = _crystal(dict(case, T=0.0), gen, dev)
        sig = 0.05 * math.sqrt(case["T"] / 300.0)
        s.x = [torch.remainder(x + sig * torch.randn(x.shape, generator=gen, device=dev, dtype=torch.float64),
                               torch.tensor(s.box, device=dev)).cpu().numpy() for _ in range(case["snapshots"])]
        s.nep = NEP(load_model(_TEACHER), lj=False)
        return s
    x, box = _crystal(case, gen, dev)
    if s.path == "noalloc":
        s.x, s.box = x.contiguous(), np.ascontiguousarray(box)
        s.params, s.keep = _c_params(load_model(_TEACHER))
        s.E = torch.zeros(1, dtype=torch.float64, device=dev)
        s.F = torch.zeros_like(s.x)
        s.W = torch.zeros(9, dtype=torch.float64, device=dev)
        return s
    s.nep, mass = _handle(case["form"])
    v = _velocities(x.shape[0], case["T"], mass, gen, dev)
    torch.cuda.synchronize()
    s.nep.set_state(x, v, box)
    s.box = box
    if s.path == "md":
        s.x, s.v = torch.empty_like(x), torch.empty_like(v)
        s.nep.compute(forces=False)
    else:
        s.x, s.v = (torch.empty(x.shape, dtype=torch.float64, pin_memory=True) for _ in range(2))
        s.nep.compute(forces=False)
        s.nep.get_state(s.x, s.v)
    return s


def _handle(form):
    teacher, student = load_model(_TEACHER), load_model(_STUDENT)
    if form in ("plain", "mix_bf16", "mix_fp16"):
        return NEP(teacher, rebuild_every=10, precision="fp32" if form == "plain" else form), teacher["mass_amu"]
    h = NEP(student, rebuild_every=10, precision="mix_bf16" if "bf16" in form else "fp32")
    if form != "student":
        h.set_fallback(teacher, student["q_lo"], student["q_hi"], margin=0.05, max_fraction=0.5)
    return h, student["mass_amu"]


def _c_params(m):
    keep = {k: np.ascontiguousarray(np.asarray(m[k], dtype=np.float32).ravel())
            for k in ("c_R", "c_A", "W0", "b0", "w1", "q_scale")}
    fp = lambda k: keep[k].ctypes.data_as(C.POINTER(C.c_float))  # noqa: E731
    return _nep.nep_params(m["n_max_R"], m["n_max_A"], m["basis_R"], m["basis_A"], m["l_max_3b"], m["l_max_4b"],
                           m["n_neu"], m["rc_R"], m["rc_A"], fp("c_R"), fp("c_A"), fp("W0"), fp("b0"), fp("w1"),
                           float(m.get("b1", 0.0)), fp("q_scale"), m["lj_eps"], m["lj_sigma"], m["lj_rc"],
                           m["mass_amu"], m["skin"], 0, 0, 0), keep


def _thermo(nep):
    th = nep.thermo()
    return np.array([th["pe"], th["ke"], th["temperature"], th["pressure"], *th["w_diag"]])


def run(s):
    if s.path == "md":
        s.nep.step(1.0, s.case["steps"])
        s.nep.get_state(s.x, s.v)
        return {"x": s.x, "v": s.v, "thermo": _thermo(s.nep)}
    if s.path == "roundtrip":
        s.nep.set_state(s.x, s.v, s.box)
        s.nep.step(1.0, 1)
        s.nep.get_state(s.x, s.v)
        return {"x": s.x, "v": s.v, "thermo": _thermo(s.nep)}
    if s.path == "label":
        E, F, W = [], [], []
        for x in s.x:
            s.nep.set_state(x, None, s.box)
            e, f, w = s.nep.compute()
            E.append(e), F.append(f), W.append(w)
        return {"E": np.array(E), "F": np.stack(F), "W": np.stack(W)}
    if s.path == "noalloc":
        st = _nep.lib().nep_compute_noalloc(C.byref(s.params), s.x.shape[0], s.x.data_ptr(),
                                            s.box.ctypes.data_as(C.POINTER(C.c_double)), s.E.data_ptr(),
                                            s.F.data_ptr(), s.W.data_ptr(), None)
        if st != 0:
            raise RuntimeError(f"nep_compute_noalloc: status {st}")
        return {"E": s.E, "F": s.F, "W": s.W}
    if s.path == "eval":
        with torch.no_grad():
            E, F = _st.student_ef(s.theta, s.qs, s.cells)
        return {"E": E, "F": F}
    s.t += 1
    s.theta.grad = None
    E, F = _st.student_ef(s.theta, s.qs, s.cells, 0, s.cells.n_cells)
    loss = _st.loss_fn(E, F, s.cells, 0, s.cells.n_cells)
    loss.backward()
    with torch.no_grad():
        _st.adam_step(s.theta.data, s.theta.grad, s.m, s.v, 5e-5, s.t)
    return {"E": E.detach(), "F": F.detach(), "loss": loss.detach(), "grad": s.theta.grad, "theta": s.theta.detach()}


# ---------------------------------------------------------------------------------------------------
# what a pass cannot do without

def _atoms(case):
    n = 4 * case["nx"] * case["ny"] * case["nz"] - case.get("vac", 0)
    return n - round(4.0 / A_CU ** 3 * 4.0 / 3.0 * math.pi * case["void"] ** 3) if case.get("void") else n


# float32 operations of one atom's energy and force evaluation at bulk coordination (42 radial and pair-term
# neighbours, 18 angular ones), counting each pair's geometry, basis, sums and adjoint contraction once
_FLOP = {"plain": 40.6e3, "mix_bf16": 37.0e3, "mix_fp16": 37.0e3, "student": 20.7e3, "student_fb": 20.7e3,
         "student_bf16_fb": 20.7e3}
_FLOP_TRAIN = 75e3                 # forward, directional derivatives and parameter gradient of the student
_FLOP_EVAL = 30e3


def work(case):
    p = case["path"]
    if p in ("train", "eval"):
        n = case["cells"] * 4 * 125
        # basis sums, pair displacements and neighbour indices read once (twice in training: forward and
        # directional derivatives), energies and forces written
        per = 4 * 72 + 20 * 42 + 12
        return {"bytes": n * (per * 2 + 4 * 72 if p == "train" else per), "flops": n * (_FLOP_TRAIN if p == "train" else _FLOP_EVAL)}
    n = _atoms(case)
    if p == "label":
        return {"bytes": case["snapshots"] * n * 48, "flops": case["snapshots"] * n * _FLOP["plain"]}
    if p == "noalloc":
        return {"bytes": n * 48, "flops": n * _FLOP["plain"]}
    steps = case.get("steps", 1)
    # per step: x and v read and written, forces written and read, float32 positions and the list read once
    return {"bytes": n * (steps * (96 + 24 + 24 + 32 + 4 * 54) + 96), "flops": n * steps * _FLOP[case["form"]]}


def tolerance(case):
    p = case["path"]
    if p == "train":
        return {"rel": 2e-5, "max": 1e-3}
    if p == "eval":
        return {"rel": 1e-5, "max": 1e-4}
    if p in ("label", "noalloc"):
        return {"rel": 2e-5, "max": 2e-4}
    if case["form"] in ("mix_bf16", "student_bf16_fb"):
        return {"rel": 2e-3, "max": 2e-2}
    if case["form"] == "mix_fp16":
        return {"rel": 3e-4, "max": 3e-3}
    return {"rel": 5e-6, "max": 1e-4}


# ---------------------------------------------------------------------------------------------------
# the same in 64 bits, plain torch: the definitions (two-neighbour Legendre sums, no harmonics), forces by autograd

class _Exact:
    def __init__(self, m, dev, lj=True, theta=None):
        t = lambda k, *sh: torch.tensor(np.asarray(m[k], np.float32).astype(np.float64), device=dev).reshape(*sh)  # noqa: E731
        self.nR, self.nA, self.l3, self.four = m["n_max_R"] + 1, m["n_max_A"] + 1, m["l_max_3b"], m["l_max_4b"] == 2
        nd = self.nR + self.nA * self.l3 + (self.nA if self.four else 0)
        self.rcR, self.rcA = m["rc_R"], m["rc_A"]
        self.qs = t("q_scale", nd)
        if theta is None:
            self.cR, self.cA = t("c_R", self.nR, 8), t("c_A", self.nA, 8)
            self.W0, self.b0, self.w1, self.b1 = t("W0", m["n_neu"], nd), t("b0", -1), t("w1", -1), float(np.float32(m.get("b1", 0.0)))
        else:
            shapes = [(self.nR, 8), (self.nA, 8), (m["n_neu"], nd), (m["n_neu"],), (m["n_neu"],), ()]
            parts = torch.split(theta, [max(1, int(np.prod(s))) for s in shapes])
            self.cR, self.cA, self.W0, self.b0, self.w1, self.b1 = (q.reshape(s) for q, s in zip(parts, shapes))
        self.lj = (float(np.float32(m["lj_eps"])), float(np.float32(m["lj_sigma"])), m["lj_rc"]) if lj else None

    @staticmethod
    def basis(r, rc):
        u = r / rc
        x = 2 * (u - 1) ** 2 - 1
        T = [torch.ones_like(x), x]
        for _ in range(6):
            T.append(2 * x * T[-1] - T[-2])
        fc = torch.where(r < rc, 0.5 * (1 + torch.cos(math.pi * u)), torch.zeros_like(r))
        return 0.5 * (torch.stack(T, -1) + 1) * fc[..., None]

    def descriptors(self, d, r):
        q = [self.basis(r, self.rcR).sum(1) @ self.cR.T]
        k = max(1, int((r < self.rcA).sum(1).max()))
        ra, o = torch.topk(r, min(k, r.shape[1]), dim=1, largest=False)
        u = torch.gather(d, 1, o[..., None].expand(-1, -1, 3)) / ra[..., None]
        g = self.basis(ra, self.rcA) @ self.cA.T
        c = u @ u.transpose(1, 2)
        P = [c, (3 * c ** 2 - 1) / 2, (5 * c ** 3 - 3 * c) / 2, (35 * c ** 4 - 30 * c ** 2 + 3) / 8]
        ql = torch.stack([((P[l] @ g) * g).sum(1) for l in range(self.l3)], -1)
        q.append(ql.reshape(ql.shape[0], -1))
        if self.four:
            T = torch.einsum("nka,nki,nkj->naij", g, u, u)
            T = T - torch.eye(3, device=d.device).double() * g.sum(1)[..., None, None] / 3
            q.append(torch.einsum("naij,najk,naki->na", T, T, T))
        return torch.cat(q, 1)

    def site(self, d, r, pair=True, q=None):
        q = self.descriptors(d, r) if q is None else q
        U = torch.tanh((q * self.qs) @ self.W0.T - self.b0) @ self.w1 - self.b1
        return U + self.pair(r) if pair and self.lj else U

    def pair(self, r):
        eps, sig, rc = self.lj
        s6, c6 = (sig / r) ** 6, (sig / rc) ** 6
        e = 4 * eps * (s6 ** 2 - s6) - 4 * eps * (c6 ** 2 - c6) - (r - rc) * 4 * eps * (6 * c6 - 12 * c6 ** 2) / rc
        return 0.5 * torch.where(r < rc, e, torch.zeros_like(e)).sum(1)


def _neighbours(x, L, rc):
    """Padded neighbour indices (-1 past the last) of every atom, minimum image."""
    n = x.shape[0]
    rows, step = [], max(1, (1 << 25) // n)
    for a in range(0, n, step):
        d2 = 0
        for c in range(3):
            t = x[a:a + step, None, c] - x[None, :, c]
            d2 = d2 + (t - L[c] * torch.round(t / L[c])) ** 2
        i, j = torch.nonzero(d2 < rc * rc, as_tuple=True)
        keep = i + a != j
        rows.append(torch.stack([i[keep] + a, j[keep]]))
    i, j = torch.cat(rows, 1)
    cnt = torch.bincount(i, minlength=n)
    out = torch.full((n, int(cnt.max())), -1, dtype=torch.int64, device=x.device)
    out[i, torch.arange(i.shape[0], device=x.device) - (torch.cumsum(cnt, 0) - cnt)[i]] = j
    return out


def _geometry(x, L, nb, a, b):
    j = nb[a:b]
    d = x[j.clamp_min(0)] - x[a:b, None]
    d = d - L * torch.round((d / L).detach())
    d = torch.where((j >= 0)[..., None], d, torch.tensor([1e3, 0.0, 0.0], device=x.device).double())
    return d, d.norm(dim=-1)


def _evaluate(x, L, nb, model, fallback=None, chunk=8192):
    """E, F [n, 3], W [3, 3] and (fallback: (teacher, lo, hi)) each atom's own model."""
    n, E = x.shape[0], 0.0
    F, W = torch.zeros_like(x), torch.zeros(3, 3, dtype=torch.float64, device=x.device)
    for a in range(0, n, chunk):
        b = min(n, a + chunk)
        d, _ = _geometry(x, L, nb, a, b)
        d = d.detach().requires_grad_(True)
        r = d.norm(dim=-1)
        q = model.descriptors(d, r)
        U = model.site(d, r, pair=False, q=q)
        if fallback is not None:
            teacher, lo, hi = fallback
            qt = (q * model.qs).detach()
            out = ((qt < lo) | (qt > hi)).any(1).nonzero()[:, 0]
            if out.numel():
                U = U.index_copy(0, out, teacher.site(d[out], r[out], pair=False))
        U = U + model.pair(r) if model.lj else U
        E += float(U.detach().sum())
        g, = torch.autograd.grad(U.sum(), d)
        valid = nb[a:b] >= 0
        F[a:b] += g.sum(1)
        F.index_add_(0, nb[a:b][valid], -g[valid])
        W -= torch.einsum("nki,nkj->ij", torch.where(valid[..., None], d.detach(), torch.zeros_like(d)), g)
    return E, F, W


def exact(case, seed):
    dev = torch.device("cuda")
    p = case["path"]
    if p in ("train", "eval"):
        return _exact_student(case, seed, dev)
    n = _atoms(case)
    if n > 140000 or (p == "md" and n * case["steps"] > 2_000_000):
        return None                # over about 20 seconds
    gen = _gen(seed, dev)
    teacher = _Exact(_model(_TEACHER), dev, lj=p != "label")
    if p == "label":
        x0, box = _crystal(dict(case, T=0.0), gen, dev)
        sig = 0.05 * math.sqrt(case["T"] / 300.0)
        L, E, F, W = torch.tensor(box, device=dev), [], [], []
        for _ in range(case["snapshots"]):
            x = torch.remainder(x0 + sig * torch.randn(x0.shape, generator=gen, device=dev, dtype=torch.float64), L)
            e, f, w = _evaluate(x, L, _neighbours(x, L, 5.0), teacher)
            E.append(e), F.append(f.cpu().numpy()), W.append(w.cpu().numpy())
        return {"E": np.array(E), "F": np.stack(F), "W": np.stack(W)}
    x, box = _crystal(case, gen, dev)
    L = torch.tensor(box, device=dev)
    if p == "noalloc":
        e, f, w = _evaluate(x, L, _neighbours(x, L, 5.0), teacher)
        return {"E": torch.tensor([e], dtype=torch.float64), "F": f, "W": w.reshape(9)}
    model, fb = teacher, None
    if "student" in case["form"]:
        sm = _model(_STUDENT)
        model = _Exact(sm, dev)
        if case["form"] != "student":
            lo, hi = (torch.tensor(np.asarray(sm[k], np.float32).astype(np.float64), device=dev) for k in ("q_lo", "q_hi"))
            w = 0.05 * (hi - lo)
            fb = (teacher, lo - w, hi + w)
    mass = _model(_TEACHER)["mass_amu"]
    v = _velocities(x.shape[0], case["T"], mass, gen, dev)
    nb = _neighbours(x, L, 6.0)    # 25 steps of 1 fs move no pair by as much as the 1 Angstrom beyond the cutoff
    E, F, W = _evaluate(x, L, nb, model, fb)
    for _ in range(case.get("steps", 1)):
        v = v + 0.5 * ACC / mass * F
        x = x + v
        E, F, W = _evaluate(x, L, nb, model, fb)
        v = v + 0.5 * ACC / mass * F
    ke = float(0.5 * mass * KE * (v * v).sum())
    W = W.cpu().numpy()
    th = np.array([E, ke, 2 * ke / ((3 * x.shape[0] - 3) * KB), (2 * ke + np.trace(W)) / (3 * float(np.prod(box))),
                   W[0, 0], W[1, 1], W[2, 2]])
    return {"x": torch.remainder(x, L), "v": v, "thermo": th}


def _exact_student(case, seed, dev):
    cells, E_ref, F_ref = _train_inputs(case, seed, dev)
    m = _model(_STUDENT)
    train = case["path"] == "train"
    n, nc = F_ref.shape[0], len(cells)
    if nc > 250:
        return None                # over about 20 seconds
    theta = torch.tensor(_st_pack(m), device=dev, requires_grad=train)
    model = _Exact(m, dev, lj=False, theta=theta)
    Fr = torch.tensor(F_ref.astype(np.float64), device=dev)
    E, F, loss, a = [], [], 0.0, 0
    grad = torch.zeros_like(theta)
    for c, (pos, box) in enumerate(cells):
        L = torch.tensor(np.asarray(box, np.float32).astype(np.float64), device=dev)
        # what the set holds: positions wrapped into the box, in float32
        x = torch.tensor(np.mod(pos, box).astype(np.float32).astype(np.float64), device=dev, requires_grad=True)
        nb = _neighbours(x.detach(), L, 5.0)
        e = model.site(*_geometry(x, L, nb, 0, x.shape[0]), pair=False).sum()
        g, = torch.autograd.grad(e, x, create_graph=train)
        E.append(e.detach()), F.append(-g.detach())
        if train:
            k = x.shape[0]
            part = ((e - float(E_ref[c])) / k) ** 2 / nc + 10.0 * ((-g - Fr[a:a + k]) ** 2).sum() / (3 * n)
            loss += float(part.detach())
            grad += torch.autograd.grad(part, theta)[0]
            model = _Exact(m, dev, lj=False, theta=theta)
            a += k
    out = {"E": torch.stack(E), "F": torch.cat(F)}
    if train:
        # one Adam step from zero moments: m / c1 = g, sqrt(v / c2) = |g|
        out.update(loss=np.float64(loss), grad=grad, theta=(theta - 5e-5 * grad / (grad.abs() + 1e-8)).detach())
    return out


def _st_pack(m):
    return np.concatenate([np.asarray(m[k], np.float32).astype(np.float64).reshape(-1)
                           for k in ("c_R", "c_A", "W0", "b0", "w1", "b1")])
