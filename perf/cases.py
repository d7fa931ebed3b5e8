"""What the performance of this framework is measured on: calls that users of a
NEP library make, each through the public entry points of
``paper_2607_06969_gb300.binding`` (or ``autograd``), over the sizes that the
repository's own workloads span (58 atoms to 3.7 million, one structure or a
batch of uneven ones, FP32, FP16/BF16 networks and FP64).

A case is a dict of plain values.  Its ``kind`` is the call that is timed:

  screen      list build + energies, forces, virial of new structures
  evaluate    energies, forces, virial on a list that is in hand
  md          ten velocity-Verlet steps from a snapshot, one list rebuild
  train       loss and parameter gradient of a batch, then an Adam step
  autograd    forward and backward through the torch.autograd Function
  evaluate64  FP64 energies, forces, virial
  train64     FP64 loss and parameter gradient

``exact`` restates the potential in 64 bits with torch alone.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2607_06969_gb300 import autograd as ag
from paper_2607_06969_gb300 import binding as nb
from paper_2607_06969_gb300 import inputs as inp

# The model shapes that the repository's workloads name, and two shapes
# without compiled kernels, which the generic FP32 path serves.
MODELS = {
    "small": inp.HYPER_SMALL,      # 38-30-1 with the 4-body term
    "table2": inp.HYPER_TABLE2,    # 42-50-1, 2+3-body
    "large": inp.HYPER_LARGE,      # 52-64-1 with the 4-body term
    "two_species": inp.Hyper(n_types=2, n_rad=11, n_ang=7, k_rad=10, k_ang=9, has_4body=0, n_hidden=20,
                             rc_rad=6.0, rc_ang=4.5),
    "narrow": inp.Hyper(n_types=3, n_rad=5, n_ang=3, k_rad=6, k_ang=5, has_4body=1, n_hidden=7),
}
CAP, CAP_ANG = 160, 80        # list capacities of the MD workloads (skin 1 A)
SKIN = 1.0                    # Verlet skin of the MD and evaluation cases, A
STEPS, DT = 10, 2.0           # one list period of velocity Verlet, fs
LOSS_W = (1.0, 1.0, 0.125)    # loss weights (E, F, V)
ADAM = (1e-3, 0.9, 0.999, 1e-8)
MVV_TO_EV = 103.6427          # 1 u A^2/fs^2 in eV
PACKING_RHO = 0.0325


# --------------------------------------------------------------------------
# cases
# --------------------------------------------------------------------------
def listed() -> list[dict]:
    return [
        # the smallest call: one new 58-atom structure (the smallest of the
        # operator-scaling sizes) is listed and evaluated, as in active
        # learning or a Monte Carlo move; latency and launches count
        dict(name="screen_58", kind="screen", model="small", precision=0, cfgs=1, lo=58, hi=58),
        # dozens of new structures of a data set, uneven and mostly smaller
        # than twice the cutoff, listed and evaluated in one batch
        dict(name="screen_batch_48", kind="screen", model="table2", precision=0, cfgs=48, lo=24, hi=512),
        # MD of a small cell (194 atoms, the smallest MD size), replayed from
        # a CUDA graph as such a program would
        dict(name="md_194_graph", kind="md", model="table2", precision=0, ncell=3, vacancy=0.2, graph=True),
        # ordinary MD of some thousand atoms, calls made one by one
        dict(name="md_7200", kind="md", model="small", precision=0, ncell=10, vacancy=0.2, graph=False),
        # MD of one large system, the headline workload
        dict(name="md_900k", kind="md", model="small", precision=0, ncell=50, vacancy=0.2, graph=False),
        # a batch of uneven replicas with the FP16 network
        dict(name="md_replicas_fp16", kind="md", model="small", precision=1, cfgs=48, lo=64, hi=4096,
             graph=False),
        # the largest system: 3.7 million atoms, wide network in FP16
        dict(name="evaluate_3m7_fp16", kind="evaluate", model="large", precision=1, ncell=80, vacancy=0.2),
        # a shape with no compiled kernels (two species), some thousand atoms
        dict(name="evaluate_generic", kind="evaluate", model="two_species", precision=0, ncell=11, vacancy=0.13),
        # a training step on 128 configurations of 24 to 512 atoms
        dict(name="train_128", kind="train", model="small", precision=0, cfgs=128, lo=24, hi=512),
        # fine-tuning through torch: a small batch, forward and backward
        dict(name="autograd_8", kind="autograd", model="table2", precision=0, cfgs=8, lo=58, hi=461),
        # FP64 reference evaluation of an odd-sized cell
        dict(name="evaluate64_3k", kind="evaluate64", model="small", precision=0, ncell=7, vacancy=0.11),
        # FP64 training operator on a small batch
        dict(name="train64_16", kind="train64", model="small", precision=0, cfgs=16, lo=24, hi=512),
    ]


def _log_int(rng: random.Random, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random) -> dict:
    kind = rng.choice(["screen", "evaluate", "evaluate", "md", "md", "replicas", "train", "train", "autograd",
                       "evaluate64", "train64", "generic"])
    vac = round(rng.uniform(0.0, 0.25), 3)
    model = rng.choice(["small", "table2", "large"])
    prec = rng.choice([0, 0, 1, 2])
    if kind == "screen":
        lo = rng.randint(24, 96)
        return dict(kind="screen", model=model, precision=0, cfgs=_log_int(rng, 1, 64), lo=lo,
                    hi=rng.randint(lo, 700))
    if kind == "evaluate":
        # 200 to 3.5 million atoms, uniform in the logarithm
        ncell = int(round(math.exp(rng.uniform(math.log(3), math.log(78)))))
        return dict(kind="evaluate", model=model, precision=prec, ncell=ncell, vacancy=vac)
    if kind == "md":
        # up to 0.8 million atoms (the larger models: 0.37 million)
        top = 46 if model == "small" and not prec else 36
        ncell = int(round(math.exp(rng.uniform(math.log(3), math.log(top)))))
        return dict(kind="md", model=model, precision=prec, ncell=ncell, vacancy=vac,
                    graph=ncell <= 12 and rng.random() < 0.5)
    if kind == "replicas":
        lo = _log_int(rng, 40, 400)
        return dict(kind="md", model=rng.choice(["small", "table2"]), precision=rng.choice([0, 1]),
                    cfgs=rng.randint(4, 48), lo=lo, hi=_log_int(rng, lo + 1, 4096), graph=False)
    if kind == "train":
        lo = rng.randint(20, 80)
        return dict(kind="train", model=model, precision=0, cfgs=_log_int(rng, 1, 96), lo=lo,
                    hi=rng.randint(lo, 512))
    if kind == "autograd":
        lo = rng.randint(20, 80)
        return dict(kind="autograd", model=model, precision=0, cfgs=_log_int(rng, 1, 32), lo=lo,
                    hi=rng.randint(lo, 512))
    if kind == "evaluate64":
        return dict(kind="evaluate64", model=rng.choice(["small", "table2", "large", "two_species", "narrow"]),
                    precision=0, ncell=rng.randint(3, 9), vacancy=vac)
    if kind == "train64":
        lo = rng.randint(20, 60)
        return dict(kind="train64", model=model, precision=0, cfgs=_log_int(rng, 1, 16), lo=lo,
                    hi=rng.randint(lo, 400))
    ncell = int(round(math.exp(rng.uniform(math.log(3), math.log(20)))))
    return dict(kind="evaluate", model=rng.choice(["two_species", "narrow"]), precision=0, ncell=ncell, vacancy=vac)


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _counts(case: dict) -> np.ndarray:
    """Atoms per configuration: the quantiles of a log-uniform distribution on
    [lo, hi], shuffled; the same for every seed."""
    n = case["cfgs"]
    q = (np.arange(n) + 0.5) / n
    c = np.round(case["lo"] * (case["hi"] / case["lo"]) ** q).astype(np.int64)
    return np.random.default_rng(1).permutation(c)


def _structure(case: dict, seed: int) -> inp.System:
    """Rock-salt cells with vacancies (ncell), or random packings (cfgs)."""
    h = MODELS[case["model"]]
    if "ncell" in case:
        s = inp.rocksalt(case["ncell"], vacancy=case["vacancy"], seed=seed)
        # the lattice planes a quarter cell away from the box faces
        s.pos = (s.pos + 1.5) % s.box[0]
    else:
        s = inp.packing_batch(_counts(case), density=PACKING_RHO, seed=seed)
    if h.n_types < 3:
        s.types = (s.types % h.n_types).astype(np.int32)
    return s


def _params(case: dict, seed: int) -> np.ndarray:
    return inp.init_params(MODELS[case["model"]], seed=seed + 1).astype(np.float32)


def _labels(case: dict, s: inp.System, seed: int):
    """Labels (E [B], F [N,3], V [B,9]) of an early training stage: residuals
    of the size of the values themselves."""
    rng = np.random.default_rng([seed, 7])
    n = np.diff(s.atom_off)
    e = rng.normal(0.0, 0.3, s.n_cfg) * n
    f = rng.normal(0.0, 0.5, (s.n_atoms, 3)).astype(np.float32)
    v = rng.normal(0.0, 0.5, (s.n_cfg, 9)) * n[:, None]
    return e, f, v


def _moments(case: dict, seed: int):
    """Adam moments of a run under way."""
    n = MODELS[case["model"]].n_params
    rng = np.random.default_rng([seed, 8])
    m1 = rng.normal(0.0, 0.02, n).astype(np.float32)
    m2 = (rng.uniform(0.5, 2.0, n) * 0.02 ** 2).astype(np.float32)
    return m1, m2


def _dev(x, dtype):
    return torch.from_numpy(np.ascontiguousarray(x)).to(dtype).cuda()


class _State:
    pass


def prepare(case: dict, seed: int):
    h, kind = MODELS[case["model"]], case["kind"]
    s = _structure(case, seed)
    theta = _params(case, seed)
    st = _State()
    st.case = case
    st.model = nb.Model(h, theta, precision=case["precision"])
    st.dsys = nb.DeviceSystem.from_inputs(s)
    N, B = s.n_atoms, s.n_cfg
    skin = 0.0 if kind in ("train", "train64", "autograd", "screen") else SKIN
    cap, cap_ang = (112, 56) if skin == 0.0 else (CAP, CAP_ANG)
    short = bool((s.box.min() < 2.0 * (h.rc_rad + skin) + 0.1))
    st.nl = nb.NeighborList(N, cap, cap_ang, shifts=short)
    st.ws = nb.Workspace(st.model, N, B, cap, cap_ang)
    if kind == "screen":
        st.out = _out(N, B, torch.float32)
        return st
    nb.neighbors(st.model, st.dsys, st.nl, skin, st.ws)
    if nb.check_list(st.nl) != nb.NEP_OK:
        raise nb.NepError(nb.check_list(st.nl), "neighbours", nb.last_error())
    if kind == "evaluate":
        st.out = _out(N, B, torch.float32)
    elif kind == "evaluate64":
        st.ws = nb.Workspace64(st.model, N, B)
        st.out = _out(N, B, torch.float64)
    elif kind == "md":
        st.masses = inp.MASSES[:h.n_types].astype(np.float32)
        vel = inp.maxwell_boltzmann(s.types, 900.0, seed=seed, atom_off=s.atom_off).astype(np.float32)
        _, force, st.e, st.v = nb.energy_forces_virial(st.model, st.dsys, st.nl, st.ws)
        st.start = (st.dsys.pos.clone(), _dev(vel.T, torch.float32), force)
        st.vel, st.force = torch.empty_like(force), torch.empty_like(force)
        st.graph = None
        if case["graph"]:
            _md(st)
            torch.cuda.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                _md(st)
            st.graph = g
    else:
        e, f, v = _labels(case, s, seed)
        st.ftype = torch.float64 if kind == "train64" else torch.float32
        st.labels = (_dev(e, torch.float64), _dev(f.T, st.ftype), _dev(v, torch.float64))
        if kind == "train64":
            st.ws = nb.Workspace64(st.model, N, B, train=True)
        else:
            st.ws = nb.Workspace(st.model, N, B, cap, cap_ang, train=True)
        st.grad = torch.empty(h.n_params, dtype=st.ftype, device="cuda")
        st.loss = torch.empty(1, dtype=torch.float64, device="cuda")
        if kind == "train":
            m1, m2 = _moments(case, seed)
            st.m1, st.m2, st.t = _dev(m1, torch.float32), _dev(m2, torch.float32), 100
        elif kind == "autograd":
            st.params = _dev(theta, torch.float32).requires_grad_(True)
            fwd = nb.Workspace(st.model, N, B, cap, cap_ang)
            st.runner = ag.NepRunner(st.model, st.dsys, st.nl, fwd, st.ws)
            n = torch.from_numpy(np.diff(s.atom_off)).double().cuda()
            st.cfg = torch.from_numpy(s.cfg_of_atom()).cuda()
            st.inv_n = 1.0 / n
    return st


def _out(N: int, B: int, dtype):
    return (torch.empty(N, dtype=dtype, device="cuda"), torch.empty(3, N, dtype=dtype, device="cuda"),
            torch.empty(B, dtype=torch.float64, device="cuda"),
            torch.empty(B, 9, dtype=torch.float64, device="cuda"))


def _md(st) -> None:
    """Ten steps from the snapshot, the list rebuilt at the first."""
    pos, vel, force = st.start
    st.dsys.pos.copy_(pos)
    st.vel.copy_(vel)
    st.force.copy_(force)
    for k in range(STEPS):
        nb.md_step(st.model, st.dsys, st.nl, st.vel, st.force, st.e, st.v, st.masses, DT, SKIN, k == 0, st.ws)


def _torch_loss(e, f, v, labels, cfg, inv_n):
    """The loss of the autograd case, written by the user in torch: per
    configuration the squared errors per atom, averaged over the batch."""
    el, fl, vl = labels
    w = LOSS_W
    per = w[0] * ((e - el) * inv_n) ** 2 + w[2] / 9.0 * (((v - vl) * inv_n[:, None]) ** 2).sum(1)
    ff = ((f - fl) ** 2).sum(0)
    return (per.sum() + (w[1] / 3.0) * (ff * inv_n.to(ff.dtype)[cfg]).sum()) / e.numel()


def run(st):
    kind = st.case["kind"]
    if kind == "screen":
        nb.neighbors(st.model, st.dsys, st.nl, 0.0, st.ws)
        return nb.energy_forces_virial(st.model, st.dsys, st.nl, st.ws, out=st.out)
    if kind == "evaluate":
        return nb.energy_forces_virial(st.model, st.dsys, st.nl, st.ws, out=st.out)
    if kind == "evaluate64":
        return nb.energy_forces_virial_fp64(st.model, st.dsys, st.nl, st.ws, out=st.out)
    if kind == "md":
        if st.graph is not None:
            st.graph.replay()
        else:
            _md(st)
        return [st.dsys.pos, st.vel, st.force, st.e, st.v]
    if kind == "train":
        nb.param_grad(st.model, st.dsys, st.nl, st.ws, *st.labels, w=LOSS_W, grad=st.grad, loss=st.loss)
        nb.adam_step(st.model, st.grad, st.m1, st.m2, st.t, *ADAM)
        st.t += 1
        return [st.grad, st.loss, st.m1, st.m2]
    if kind == "train64":
        return list(nb.param_grad_fp64(st.model, st.dsys, st.nl, st.ws, *st.labels, w=LOSS_W, grad=st.grad,
                                       loss=st.loss))
    st.params.grad = None
    e, f, v = ag.energy_forces_virial(st.params, st.runner)
    loss = _torch_loss(e, f, v, st.labels, st.cfg, st.inv_n)
    loss.backward()
    return [e, f, v, loss, st.params.grad]


# --------------------------------------------------------------------------
# work and tolerance
# --------------------------------------------------------------------------
def _atoms(case: dict) -> int:
    if "ncell" in case:
        cations = 4 * case["ncell"] ** 3
        return 2 * cations - int(round(case["vacancy"] * cations))
    return int(_counts(case).sum())


def work(case: dict) -> dict:
    """Operations of the formulas (FMA = 2) with the neighbours inside the
    cutoffs; bytes: positions, species and list in, results out."""
    h, kind = MODELS[case["model"]], case["kind"]
    N = _atoms(case)
    rho = (8.0 - 4.0 * case["vacancy"]) / 216.0 if "ncell" in case else PACKING_RHO
    nr = rho * 4.0 / 3.0 * math.pi * h.rc_rad ** 3
    na = rho * 4.0 / 3.0 * math.pi * h.rc_ang ** 3
    K, Ka, nA, D, H = h.k_rad, h.k_ang, h.n_ang, h.dim, h.n_hidden
    basis, basis_d = (lambda k: 8 + 5 * (k - 1)), (lambda k: 20 + 13 * (k - 2))
    evaluation = (nr * (21 + basis(K) + 2 * K) + 4 * h.n_rad * h.n_types * K
                  + na * (10 + basis(Ka) + 2 * nA * Ka + 45 + 48 * nA) + 244 * nA + H * (4 * D + 6)
                  + na * (10 + basis_d(Ka) + 4 * nA * Ka + 45 + 96 * nA + 276)
                  + nr * (52 + basis_d(K) + 4 * K))
    real = 8 if kind.endswith("64") else 4
    per_eval = N * (16 + 4 * nr + 4 * real)          # pos, type, list; force, energy
    if kind in ("screen", "evaluate", "evaluate64"):
        extra = N * (4 * nr + 4) if kind == "screen" else 0
        return dict(bytes=float(per_eval + extra), flops=float(N * evaluation))
    if kind == "md":
        # per step also velocities in and out, positions and forces in and out
        return dict(bytes=float(STEPS * (per_eval + 48 * N)), flops=float(STEPS * N * evaluation))
    # the tangent of the descriptors, the network's second-order terms, the
    # angular pair coefficients, and four operations per atom and parameter of
    # its species
    backward = (nr * (60 + basis_d(K) + 2 * K) + na * (2 * (45 + basis_d(Ka)) + 8 * nA * Ka + 24 * 16 + 240 * nA)
                + H * (6 * D + 12) + 4 * h.n_params / h.n_types)
    return dict(bytes=float(per_eval + N * 3 * real + 4 * 8 * h.n_params), flops=float(N * (evaluation + backward)))


def tolerance(case: dict) -> dict:
    """About four times what was seen against 64 bits.  FP32: 3e-6 in one
    evaluation and 7e-7 in a gradient; over ten steps of MD the positions'
    own rounding gives 2e-5 in the forces and grows with the box.  FP16 and
    BF16 networks: 3e-4 in forces and energies, but 1e-2 in the virials, whose
    sums cancel."""
    kind = case["kind"]
    if kind.endswith("64"):
        return dict(rel=1e-12, max=1e-10)
    if case["precision"]:
        return dict(rel=0.03 if case["precision"] == 2 else 0.015, max=0.5)
    return dict(rel=1e-4, max=4e-3) if kind == "md" else dict(rel=1e-5, max=1e-3)


# --------------------------------------------------------------------------
# the same quantities in 64 bits, torch alone
# --------------------------------------------------------------------------
def _harmonic_table():
    """(l, m, polynomial coefficients of d^m P_l / dz^m, weight): real
    harmonics T with sum_m T(a) T(b) = P_l(a . b)."""
    out = []
    for l in range(1, 5):
        p = np.polynomial.legendre.leg2poly([0.0] * l + [1.0])
        for m in range(l + 1):
            c = np.polynomial.polynomial.polyder(p, m) if m else p
            w = 1.0 if m == 0 else 2.0 * math.factorial(l - m) / math.factorial(l + m)
            out.append((l, m, [float(x) for x in c], math.sqrt(w)))
    return out


_HARMONICS = _harmonic_table()
_L_OF = [l for l, m, _, _ in _HARMONICS for _ in range(1 if m == 0 else 2)]


def _harmonics(u):
    x, y, z = u.unbind(1)
    re, im = [torch.ones_like(x)], [torch.zeros_like(x)]
    for _ in range(4):                              # (x + iy)^m
        re.append(re[-1] * x - im[-1] * y)
        im.append(re[-2] * y + im[-1] * x)
    cols = []
    for _, m, c, w in _HARMONICS:
        p = torch.full_like(z, c[-1])
        for a in reversed(c[:-1]):
            p = p * z + a
        p = p * w
        cols += [p * re[m]] if m == 0 else [p * re[m], p * im[m]]
    return torch.stack(cols, 1)


def _basis(r, rc, K):
    x = 2.0 * (r / rc - 1.0) ** 2 - 1.0
    fc = 0.5 * (1.0 + torch.cos(math.pi * r / rc))
    t = [torch.ones_like(x), x]
    while len(t) < K:
        t.append(2.0 * x * t[-1] - t[-2])
    return torch.stack([0.5 * (a + 1.0) * fc for a in t[:K]], 1)


def _unpack(h, theta):
    D, H, T = h.dim, h.n_hidden, h.n_types
    n = H * D + 2 * H + 1
    mlp = theta[:T * n].view(T, n)
    W0, b0 = mlp[:, :H * D].view(T, H, D), mlp[:, H * D:H * D + H]
    w1, b1 = mlp[:, H * D + H:H * D + 2 * H], mlp[:, -1]
    nR = T * T * h.n_rad * h.k_rad
    cR = theta[T * n:T * n + nR].view(T, T, h.n_rad, h.k_rad)
    cA = theta[T * n + nR:].view(T, T, h.n_ang, h.k_ang)
    return W0, b0, w1, b1, cR, cA


def _energies(h, prm, ti, i, tj, d):
    """E of the centres with species ti; pairs (centre i, species tj, r_ij)."""
    W0, b0, w1, b1, cR, cA = prm
    n, T = ti.numel(), h.n_types
    r = d.norm(dim=1)
    F = torch.zeros(n * T, h.k_rad, dtype=d.dtype, device=d.device)
    F = F.index_add(0, i * T + tj, _basis(r, h.rc_rad, h.k_rad))
    q = [torch.einsum("atnk,atk->an", cR[ti], F.view(n, T, -1))]
    near = torch.nonzero(r < h.rc_ang).squeeze(1)
    da, ra = d[near], r[near]
    u = da / ra[:, None]
    Q = _basis(ra, h.rc_ang, h.k_ang)
    idx = i[near] * T + tj[near]

    def sums(Y):                                    # sum_j g_n(r_ij) Y(u_ij)
        m = Y.shape[1]
        z = torch.zeros(n * T, h.k_ang * m, dtype=d.dtype, device=d.device)
        z = z.index_add(0, idx, (Q[:, :, None] * Y[:, None, :]).flatten(1))
        return torch.einsum("atnk,atkm->anm", cA[ti], z.view(n, T, h.k_ang, m))

    S2 = sums(_harmonics(u)) ** 2
    ql = torch.stack([S2[:, :, [c for c, l in enumerate(_L_OF) if l == k]].sum(2) for k in range(1, 5)], 2)
    q.append(ql.flatten(1))
    if h.has_4body:
        x, y, z = u.unbind(1)
        M = sums(torch.stack([x * x, x * y, x * z, y * y, y * z, z * z], 1))
        A = M[:, :, [0, 1, 2, 1, 3, 4, 2, 4, 5]].view(n, h.n_ang, 3, 3)
        A = A - torch.eye(3, dtype=d.dtype, device=d.device) * (A.diagonal(dim1=2, dim2=3).sum(2) / 3.0)[..., None, None]
        q.append((A @ A @ A).diagonal(dim1=2, dim2=3).sum(2))
    q = torch.cat(q, 1)
    E = torch.zeros(n, dtype=d.dtype, device=d.device)
    for t in range(T):
        at = torch.nonzero(ti == t).squeeze(1)
        hid = torch.tanh(q[at] @ W0[t].T + b0[t])
        E = E.index_add(0, at, hid @ w1[t] + b1[t])
    return E


def _pairs_small(pos, a0, a1, L, rc):
    """All (i, j, image) of one configuration inside rc, by trial."""
    p = pos[a0:a1]
    n = a1 - a0
    reach = [int(math.ceil(rc / float(x))) for x in L]
    whole = all(float(x) > 2.0 * rc for x in L)
    imgs = [(0, 0, 0)] if whole else [(x, y, z) for x in range(-reach[0], reach[0] + 1)
                                      for y in range(-reach[1], reach[1] + 1)
                                      for z in range(-reach[2], reach[2] + 1)]
    S = torch.tensor(imgs, dtype=torch.float64, device=pos.device) * L
    rows = max(1, int(2e7 / (n * len(imgs))))
    I, J, D = [], [], []
    for c0 in range(0, n, rows):
        c1 = min(n, c0 + rows)
        d = p[None, :, :] - p[c0:c1, None, :]
        if whole:
            d = (d - L * torch.round(d / L))[:, :, None, :]
        else:
            d = d[:, :, None, :] + S
        r2 = (d * d).sum(3)
        ok = (r2 < rc * rc) & (r2 > 1e-12)
        w = torch.nonzero(ok)
        I.append(w[:, 0] + a0 + c0)
        J.append(w[:, 1] + a0)
        D.append(d[ok])
    return torch.cat(I), torch.cat(J), torch.cat(D)


def _pairs_large(pos, L, rc, rows=16384):
    """The same for one large configuration, through cells of edge >= rc, as
    chunks of centres (which come in cell order)."""
    nc = [max(3, int(float(x) / rc)) for x in L]
    c = torch.minimum((pos / L * torch.tensor(nc, device=pos.device)).long(), torch.tensor(nc, device=pos.device) - 1)
    cell = (c[:, 0] * nc[1] + c[:, 1]) * nc[2] + c[:, 2]
    order = torch.argsort(cell)
    count = torch.bincount(cell, minlength=nc[0] * nc[1] * nc[2])
    first = torch.cumsum(count, 0) - count
    most = int(count.max())
    off = torch.tensor([(x, y, z) for x in (-1, 0, 1) for y in (-1, 0, 1) for z in (-1, 0, 1)], device=pos.device)
    lane = torch.arange(most, device=pos.device)
    size = torch.tensor(nc, device=pos.device)
    for c0 in range(0, pos.shape[0], rows):
        i = order[c0:c0 + rows]
        w = (c[i][:, None, :] + off) % size
        w = (w[..., 0] * nc[1] + w[..., 1]) * nc[2] + w[..., 2]
        j = first[w][..., None] + lane
        ok = (lane < count[w][..., None]).flatten(1)
        j = order[j.flatten(1).clamp(max=pos.shape[0] - 1)]
        d = pos[j] - pos[i][:, None, :]
        d = d - L * torch.round(d / L)
        r2 = (d * d).sum(2)
        ok &= (r2 < rc * rc) & (r2 > 1e-12)
        at = torch.nonzero(ok)
        yield i[at[:, 0]], j[ok], d[ok]


def _pair_chunks(s, pos, box, rc):
    """(i, j, r_ij) with every centre's pairs in one chunk."""
    if s.n_cfg == 1 and s.n_atoms > 20000:
        yield from _pairs_large(pos, box[0], rc)
        return
    I, J, D, have = [], [], [], 0
    for b in range(s.n_cfg):
        a0, a1 = int(s.atom_off[b]), int(s.atom_off[b + 1])
        i, j, d = _pairs_small(pos, a0, a1, box[b], rc)
        I.append(i), J.append(j), D.append(d)
        have += a1 - a0
        if have > 8000 or b == s.n_cfg - 1:
            yield torch.cat(I), torch.cat(J), torch.cat(D)
            I, J, D, have = [], [], [], 0


def _evaluate(h, prm, s, pos, types, cfg, box, graph=False):
    """(E_i, F, E_b, V_b) in 64 bits; graph keeps the parameter derivatives."""
    N, B = s.n_atoms, s.n_cfg
    z = dict(dtype=torch.float64, device=pos.device)
    e, f, v = torch.zeros(N, **z), torch.zeros(N, 3, **z), torch.zeros(B, 9, **z)
    for i, j, d in _pair_chunks(s, pos, box, h.rc_rad):
        d = d.detach().requires_grad_(True)
        here, local = torch.unique(i, return_inverse=True)
        E = _energies(h, prm, types[here], local, types[j], d)
        g, = torch.autograd.grad(E.sum(), d, create_graph=graph)
        if not graph:
            E, d = E.detach(), d.detach()
        e = e.index_add(0, here, E)
        f = f.index_add(0, i, g).index_add(0, j, -g)
        v = v.index_add(0, cfg[i], -(g[:, :, None] * d[:, None, :]).flatten(1))
    lone = torch.ones(N, dtype=torch.bool, device=pos.device)   # atoms with no neighbour at all
    for i, _, _ in _pair_chunks(s, pos, box, h.rc_rad):
        lone[i] = False
    if bool(lone.any()):
        at = torch.nonzero(lone).squeeze(1)
        none = torch.zeros(0, dtype=torch.long, device=pos.device)
        e = e.index_add(0, at, _energies(h, prm, types[at], none, none, torch.zeros(0, 3, **z)))
    return e, f, torch.zeros(B, **z).index_add(0, cfg, e), v


def exact(case: dict, seed: int):
    if _atoms(case) > 1_000_000:
        return None                                 # would take too long
    h, kind = MODELS[case["model"]], case["kind"]
    s = _structure(case, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    put = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(dev)   # noqa: E731
    pos, box = put(s.pos32()).double(), put(s.box.astype(np.float32)).double()
    types, cfg = put(s.types).long(), put(s.cfg_of_atom())
    theta = put(_params(case, seed)).double()
    if kind in ("screen", "evaluate", "evaluate64"):
        e, f, et, v = _evaluate(h, _unpack(h, theta), s, pos, types, cfg, box)
        return e, f.T, et, v
    if kind == "md":
        if _atoms(case) > 100_000:
            return None                             # ten large evaluations take too long
        prm = _unpack(h, theta)
        vel = put(inp.maxwell_boltzmann(s.types, 900.0, seed=seed, atom_off=s.atom_off).astype(np.float32)).double()
        im = 1.0 / (put(inp.MASSES.astype(np.float32)).double()[types] * MVV_TO_EV)
        L = box[cfg]
        _, f, et, v = _evaluate(h, prm, s, pos, types, cfg, box)
        for k in range(STEPS):
            vel = vel + 0.5 * DT * f * im[:, None]
            pos = pos + DT * vel
            if k == 0:
                pos = pos - L * torch.floor(pos / L)
            _, f, et, v = _evaluate(h, prm, s, pos - L * torch.floor(pos / L), types, cfg, box)
            vel = vel + 0.5 * DT * f * im[:, None]
        return [pos.T, vel.T, f.T, et, v]
    labels = [put(x).double() for x in _labels(case, s, seed)]
    theta.requires_grad_(True)
    e, f, et, v = _evaluate(h, _unpack(h, theta), s, pos, types, cfg, box, graph=True)
    n = torch.bincount(cfg, minlength=s.n_cfg).double()
    loss = _torch_loss(et, f.T, v, (labels[0], labels[1].T, labels[2]), cfg, 1.0 / n)
    grad, = torch.autograd.grad(loss, theta)
    loss = loss.detach()
    if kind == "autograd":
        return [et.detach(), f.detach().T, v.detach(), loss, grad]
    if kind == "train64":
        return [grad, loss.reshape(1)]
    m1, m2 = (put(x).double() for x in _moments(case, seed))
    _, b1, b2, _ = ADAM
    return [grad, loss.reshape(1), b1 * m1 + (1 - b1) * grad, b2 * m2 + (1 - b2) * grad * grad]
