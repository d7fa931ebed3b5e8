"""Kernels whose work is split differently by system size, at the sizes where
a split can go wrong: chunk and tile edges, remainders, the smallest systems
and both sides of each dispatch rule."""
import numpy as np
import pytest

from paper_2607_06969_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nb():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2607_06969_gb300 import build as B
    B.build()
    from paper_2607_06969_gb300 import binding
    binding.lib()
    return binding


def setup(nb, h, counts, tag, skin=0.0, cap=128, cap_ang=64, seed=5, precision=0):
    s = I.packing_batch(counts, tag=tag)
    s.box[np.diff(s.atom_off) == 0] = 20.0          # an empty configuration still has a box
    model = nb.Model(h, I.init_params(h, seed=seed).astype(np.float32), precision=precision)
    dsys = nb.DeviceSystem.from_inputs(s)
    nl = nb.NeighborList(s.n_atoms, cap, cap_ang)
    ws = nb.Workspace(model, s.n_atoms, s.n_cfg, cap, cap_ang)
    nb.neighbors(model, dsys, nl, skin, ws)
    assert nb.check_list(nl) == nb.NEP_OK, nb.last_error()
    return s, model, dsys, nl, ws


@pytest.mark.parametrize("counts", [[1024], [1023, 1], [1000, 25], [2047, 2]])
def test_fp64_gradient_chunk_edges(nb, counts):
    """The gradient is linear in its adjoints, so that of a batch is the sum
    of those of its configurations: the 1,024-atom chunks of the batch fall
    elsewhere than those of the configurations.  About 10^5 terms a
    parameter, each rounded in double: 1e-12 of the largest."""
    import torch
    h = I.Hyper(n_rad=5, n_ang=3, k_rad=6, k_ang=5, n_hidden=7)   # no count a multiple of its item's block
    s, model, dsys, nl, _ = setup(nb, h, counts, 61)
    rng = np.random.default_rng(3)
    lam = rng.normal(size=(3, s.n_atoms))
    a_e, mu = rng.normal(size=s.n_cfg), rng.normal(size=(s.n_cfg, 9))

    def grad(dsys, nl, lo, hi, b0, b1):
        ws = nb.Workspace64(model, dsys.n_atoms, dsys.n_cfg, train=True)
        dev = dict(dtype=torch.float64, device="cuda")
        return nb.param_grad_adjoint_fp64(
            model, dsys, nl, ws, torch.tensor(a_e[b0:b1], **dev),
            torch.tensor(np.ascontiguousarray(lam[:, lo:hi]), **dev), torch.tensor(mu[b0:b1], **dev)).cpu().numpy()

    whole = grad(dsys, nl, 0, s.n_atoms, 0, s.n_cfg)
    total = np.zeros_like(whole)
    for b in range(s.n_cfg):
        lo, hi = int(s.atom_off[b]), int(s.atom_off[b + 1])
        sub = I.System(pos=s.pos[lo:hi], types=s.types[lo:hi], box=s.box[b:b + 1], atom_off=np.array([0, hi - lo]))
        d2 = nb.DeviceSystem.from_inputs(sub)
        n2 = nb.NeighborList(sub.n_atoms, 128, 64)
        w2 = nb.Workspace(model, sub.n_atoms, 1, 128, 64)
        nb.neighbors(model, d2, n2, 0.0, w2)
        total += grad(d2, n2, lo, hi, b, b + 1)
    assert np.abs(whole - total).max() <= 1e-12 * np.abs(total).max()
    # d/db1 of a species is the sum of a_e over its atoms
    assert np.isfinite(whole).all()
    for t in range(h.n_types):
        at = (t + 1) * (h.n_hidden * h.dim + 2 * h.n_hidden + 1) - 1
        want = a_e[s.cfg_of_atom()][s.types == t].sum()
        assert abs(whole[at] - want) <= 1e-10 * s.n_atoms


MODELS = dict(small=I.HYPER_SMALL, table2=I.HYPER_TABLE2, large=I.HYPER_LARGE,
              tiny=I.Hyper(n_rad=3, n_ang=2, k_rad=4, k_ang=3, n_hidden=5, rc_rad=5.0, rc_ang=4.0))


def both_forms(nb, model, dsys, nl, ws):
    """(default choice, one thread per atom) of one evaluation, as arrays."""
    got = [t.cpu().numpy().copy() for t in nb.energy_forces_virial(model, dsys, nl, ws)]
    nb.set_variant(model, 0)
    want = [t.cpu().numpy().copy() for t in nb.energy_forces_virial(model, dsys, nl, ws)]
    nb.set_variant(model, -1)
    again = [t.cpu().numpy().copy() for t in nb.energy_forces_virial(model, dsys, nl, ws)]
    for x, y in zip(got, again):
        assert np.array_equal(x, y)
    return got, want


def assert_close(got, want, n, tol=1.0):
    """FP32 sums of some tens of terms of order 0.1 to 1 in another order:
    1e-6 eV in E_i, 1e-5 eV/A in the forces, and per atom in the totals."""
    assert np.abs(got[0] - want[0]).max() <= tol * 1e-6
    assert np.abs(got[1] - want[1]).max() <= tol * 1e-5
    assert np.all(np.abs(got[2] - want[2]) <= tol * 1e-6 * np.maximum(n, 1))
    assert np.all(np.abs(got[3] - want[3]).max(1) <= tol * 1e-5 * np.maximum(n, 1))


@pytest.mark.parametrize("hname", list(MODELS))
@pytest.mark.parametrize("counts,skin", [([1], 0.0), ([3], 0.0), ([2, 0, 33], 0.5), ([24, 127, 130], 1.0),
                                         ([1500, 1499], 0.0), ([1500, 1501], 0.0), ([3700, 17, 300], 1.0),
                                         ([3701], 0.5), ([8000], 0.0), ([8001], 0.0),
                                         ([6000, 4000], 0.5), ([6000, 4001], 0.5), ([6000, 4001, 2], 0.0)])
def test_lane_groups_agree_with_one_thread_per_atom(nb, hname, counts, skin):
    """A group of lanes per atom (32 up to 3,000 atoms, then 8, the finish 16 up
    to 8,000 without images; above 10,000 for the radial sums and the finish
    only): fewer atoms than one block holds, remainders of a block, an empty
    configuration, both sides of the lines between the forms, boxes shorter
    than the cutoff (images) and longer, with a skin."""
    h = MODELS[hname]
    s, model, dsys, nl, ws = setup(nb, h, counts, 62, skin=skin, cap=160, cap_ang=80)
    assert_close(*both_forms(nb, model, dsys, nl, ws), np.diff(s.atom_off))


def test_lane_groups_many_angular_pairs(nb):
    """More angular pairs per atom than the group's slot list holds (96)."""
    s = I.packing_batch([500, 40], density=0.25, dmin=1.1, tag=63)
    h = I.HYPER_SMALL
    model = nb.Model(h, I.init_params(h, seed=5).astype(np.float32))
    dsys = nb.DeviceSystem.from_inputs(s)
    nl = nb.NeighborList(s.n_atoms, 640, 256)
    ws = nb.Workspace(model, s.n_atoms, s.n_cfg, 640, 256)
    nb.neighbors(model, dsys, nl, 0.0, ws)
    assert nb.check_list(nl) == nb.NEP_OK, nb.last_error()
    assert int(nl.cnt_ang.max()) > 96
    got, want = both_forms(nb, model, dsys, nl, ws)
    # six to seven times the pairs of the normal density, and sums as much larger
    scale = max(1.0, float(np.abs(want[1]).max()))
    assert_close(got, want, np.diff(s.atom_off), tol=10.0 * scale)


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("hname", ["small", "table2", "large"])
def test_lane_groups_16bit_network(nb, hname, precision):
    """The 16-bit network of the group form rounds q, W0 and g as the tensor-
    core kernel does: the two differ only where FP32 sums in another order put
    an operand on the other side of a rounding step (2^-11 or 2^-8 of it, one
    operand in about a thousand), far below the 16-bit error itself."""
    h = MODELS[hname]
    s, model, dsys, nl, ws = setup(nb, h, [130, 77], 64, precision=precision)
    got, want = both_forms(nb, model, dsys, nl, ws)
    step = 2.0 ** -11 if precision == 1 else 2.0 ** -8
    assert np.abs(got[0] - want[0]).max() <= 0.5 * step
    assert np.sqrt(np.mean((got[1] - want[1]) ** 2)) <= 0.1 * step


@pytest.mark.parametrize("n,L,skin,copies", [(3, 5.0, 1.0, 30000), (58, 0.0, 0.0, 1500), (700, 0.0, 1.0, 120),
                                             (8190, 0.0, 0.5, 12), (8200, 0.0, 0.5, 12),
                                             (540, 12.93, 0.0, 140)])
def test_list_build_small_and_large_forms_agree(nb, n, L, skin, copies):
    """A configuration listed alone (binned by one CTA up to 8,192 atoms, a
    warp per atom in the build and the reverse search) gets, entry for entry,
    the list of each of its copies in a batch large enough for one thread per
    atom: a few atoms in a box shorter than the cutoff (stencils too large for
    the row table), boxes with images and without, a dense one with more hits
    per atom than the warp keeps (192)."""
    h = I.HYPER_SMALL
    dense = L > 10
    s = I.packing_batch([n], tag=65, dmin=1.1 if dense else 1.5 if L else 2.4, density=n / L ** 3 if L else 0.0325)
    model = nb.Model(h, I.init_params(h).astype(np.float32))
    cap, cap_ang = (720, 250) if dense else (160, 80)

    def build(copies):
        batch = I.System(pos=np.tile(s.pos, (copies, 1)), types=np.tile(s.types, copies),
                         box=np.repeat(s.box, copies, 0), atom_off=n * np.arange(copies + 1))
        dsys = nb.DeviceSystem.from_inputs(batch)
        nl = nb.NeighborList(batch.n_atoms, cap, cap_ang)
        ws = nb.Workspace(model, batch.n_atoms, copies, cap, cap_ang)
        nb.neighbors(model, dsys, nl, skin, ws)
        assert nb.check_list(nl) == nb.NEP_OK, nb.last_error()
        get = lambda t: t.cpu().numpy().reshape(-1, batch.n_atoms)   # noqa: E731
        return [get(t) for t in (nl.cnt, nl.cnt_ang, nl.nbr, nl.rev, nl.shift)], nl.c.min_image

    one, mi = build(1)
    many, mi2 = build(copies)
    assert mi == mi2
    for c in (0, copies - 1):
        cols = slice(c * n, (c + 1) * n)
        assert np.array_equal(one[0], many[0][:, cols]) and np.array_equal(one[1], many[1][:, cols])
        used = np.arange(cap)[:, None] < one[0]
        ang = np.arange(cap_ang)[:, None] < one[1]
        assert np.array_equal(one[2][used], many[2][:, cols][used] - c * n)
        assert np.array_equal(one[3][ang], many[3][:, cols][ang])
        if not mi:
            assert np.array_equal(one[4][used], many[4][:, cols][used])


@pytest.mark.parametrize("n", [200, 480, 500, 900, 2100])
def test_first_list_of_a_process(n):
    """The one-block binning asks for its shared memory at every size that
    needs it, also when no larger system came before: each in a new process."""
    import subprocess
    import sys
    code = ("import numpy as np\nfrom paper_2607_06969_gb300 import binding as nb, inputs as I\n"
            f"s = I.packing_batch([{n}], tag=67)\nh = I.HYPER_SMALL\n"
            "m = nb.Model(h, I.init_params(h).astype(np.float32))\nd = nb.DeviceSystem.from_inputs(s)\n"
            "nl = nb.NeighborList(s.n_atoms, 128, 64)\nws = nb.Workspace(m, s.n_atoms, 1, 128, 64)\n"
            "nb.neighbors(m, d, nl, 0.0, ws)\nassert nb.check_list(nl) == nb.NEP_OK, nb.last_error()\n")
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]


@pytest.mark.parametrize("hname", list(MODELS))
@pytest.mark.parametrize("counts,skin", [([1], 0.0), ([2, 0, 3], 0.0), ([24, 127, 130], 0.7), ([900, 1101], 0.0),
                                         ([1500, 1501], 0.0)])
def test_lane_groups_training_agrees_with_one_thread_per_atom(nb, hname, counts, skin):
    """The loss gradient and the adjoint product by lane groups against the
    one-thread-per-atom kernels: remainders of a block, an empty
    configuration, each group size of forward and backward, a list with a skin.  FP32 sums
    of about 10^3 to 10^5 terms in another order: 1e-5 in relative L2 (the
    bar against the FP64 gradient is 1e-4)."""
    import torch
    h = MODELS[hname]
    s, model, dsys, nl, _ = setup(nb, h, counts, 66, skin=skin, cap=160, cap_ang=80)
    ws = nb.Workspace(model, s.n_atoms, s.n_cfg, 160, 80, train=True)
    rng = np.random.default_rng(4)
    dev = lambda x, t: torch.tensor(np.ascontiguousarray(x), dtype=t, device="cuda")   # noqa: E731
    e = dev(rng.normal(size=s.n_cfg), torch.float64)
    f = dev(rng.normal(size=(3, s.n_atoms)), torch.float32)
    v = dev(rng.normal(size=(s.n_cfg, 9)), torch.float64)

    def grads():
        g1, loss = nb.param_grad(model, dsys, nl, ws, e, f, v)
        g2 = nb.param_grad_adjoint(model, dsys, nl, ws, e, f, v)
        return g1.cpu().numpy(), loss.item(), g2.cpu().numpy()

    got = grads()
    nb.set_variant(model, 0)
    want = grads()
    nb.set_variant(model, -1)
    for x, y in zip(got, want):
        assert np.linalg.norm(np.asarray(x) - y) <= 1e-5 * np.linalg.norm(y)
    for x, y in zip(got, grads()):
        assert np.array_equal(x, y)


SHAPES64 = dict(small=I.HYPER_SMALL, large=I.HYPER_LARGE,
                narrow=I.Hyper(n_types=3, n_rad=5, n_ang=3, k_rad=6, k_ang=5, has_4body=1, n_hidden=7),
                k12=I.Hyper(n_types=2, n_rad=11, n_ang=7, k_rad=10, k_ang=9, has_4body=0, n_hidden=35),
                wide=I.Hyper(n_types=1, n_rad=16, n_ang=9, k_rad=13, k_ang=16, has_4body=1, n_hidden=33))


def typed(s, h):
    return I.System(pos=s.pos, types=(s.types % h.n_types).astype(np.int32), box=s.box, atom_off=s.atom_off)


@pytest.mark.parametrize("name", list(SHAPES64))
def test_fp64_and_generic_lane_group_sizes(nb, name):
    """The FP64 evaluation and gradient, and the generic FP32 evaluation,
    with 32 lanes per atom (up to 1,500 atoms; 4,000 generic) and with 8: a configuration
    alone against the same one in a larger batch, for shapes on every set of
    compiled loop bounds.  FP64 sums of some thousand terms: 1e-12; FP32: the
    bars of the parity tests."""
    import torch
    h = SHAPES64[name]
    one, two = I.packing_batch([43], tag=70), I.packing_batch([1470], tag=71)
    rest = I.packing_batch([3960], tag=72)
    both = I.System(pos=np.concatenate([one.pos, two.pos]), types=np.concatenate([one.types, two.types]),
                    box=np.concatenate([one.box, two.box]), atom_off=np.array([0, 43, 1513]))
    model = nb.Model(h, I.init_params(h, seed=6).astype(np.float32))
    rng = np.random.default_rng(5)
    a_e, lam, mu = rng.normal(size=2), rng.normal(size=(3, 1513)), rng.normal(size=(2, 9))
    a_e[1] = 0.0
    lam[:, 43:] = 0.0
    mu[1] = 0.0
    dev = lambda x: torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device="cuda")   # noqa: E731
    res = []
    for s, B in ((one, 1), (both, 2)):
        s = typed(s, h)
        dsys = nb.DeviceSystem.from_inputs(s)
        nl = nb.NeighborList(s.n_atoms, 160, 80)
        ws = nb.Workspace(model, s.n_atoms, B, 160, 80)
        nb.neighbors(model, dsys, nl, 0.5, ws)
        assert nb.check_list(nl) == nb.NEP_OK
        e, f, et, v = nb.energy_forces_virial_fp64(model, dsys, nl, nb.Workspace64(model, s.n_atoms, B))
        g = nb.param_grad_adjoint_fp64(model, dsys, nl, nb.Workspace64(model, s.n_atoms, B, train=True), dev(a_e[:B]),
                                       dev(lam[:, :s.n_atoms]), dev(mu[:B]))
        x = [e[:43], f[:, :43], et[:1], v[:1], g]
        y = nb.energy_forces_virial(model, dsys, nl, ws)
        res.append([t.cpu().numpy() for t in x] + [t.cpu().numpy() for t in (y[0][:43], y[1][:, :43], y[2][:1], y[3][:1])])
    for a, b in zip(res[0][:5], res[1][:5]):
        assert np.abs(a - b).max() <= 1e-12 * max(1.0, np.abs(a).max()) * 43
    s = typed(I.System(pos=np.concatenate([one.pos, rest.pos]), types=np.concatenate([one.types, rest.types]),
                       box=np.concatenate([one.box, rest.box]), atom_off=np.array([0, 43, 4003])), h)
    dsys = nb.DeviceSystem.from_inputs(s)
    nl = nb.NeighborList(s.n_atoms, 160, 80)
    ws = nb.Workspace(model, s.n_atoms, 2, 160, 80)
    nb.neighbors(model, dsys, nl, 0.5, ws)
    assert nb.check_list(nl) == nb.NEP_OK
    y = nb.energy_forces_virial(model, dsys, nl, ws)
    res.append(res[0][:5] + [t.cpu().numpy() for t in (y[0][:43], y[1][:, :43], y[2][:1], y[3][:1])])
    for got in res:                                   # the FP32 evaluation against FP64
        assert np.abs(got[5] - got[0]).max() <= 1e-6 * max(1.0, np.abs(got[0]).max())
        assert np.abs(got[6] - got[1]).max() <= 1e-4
        assert np.abs(got[8] - got[3]).max() <= 1e-5 * 43 * max(1.0, np.abs(got[3]).max())


@pytest.mark.parametrize("hname", ["small", "k12"])
def test_fp64_and_generic_many_angular_pairs(nb, hname):
    """More angular pairs than the FP64 force kernel keeps slots for (128),
    against the FP32 evaluation of the same list (its own bars, scaled with
    the forces)."""
    h = SHAPES64[hname]
    s = typed(I.packing_batch([400], density=0.32, dmin=1.0, tag=73), h)
    model = nb.Model(h, I.init_params(h, seed=5).astype(np.float32))
    dsys = nb.DeviceSystem.from_inputs(s)
    nl = nb.NeighborList(s.n_atoms, 800, 320)
    ws = nb.Workspace(model, s.n_atoms, 1, 800, 320)
    nb.neighbors(model, dsys, nl, 0.0, ws)
    assert nb.check_list(nl) == nb.NEP_OK, nb.last_error()
    assert int(nl.cnt_ang.max()) > 128
    e, f, et, v = [t.cpu().numpy() for t in nb.energy_forces_virial(model, dsys, nl, ws)]
    e6, f6, et6, v6 = [t.cpu().numpy()
                       for t in nb.energy_forces_virial_fp64(model, dsys, nl, nb.Workspace64(model, s.n_atoms, 1))]
    scale = max(1.0, float(np.abs(f6).max()))
    assert np.abs(e - e6).max() <= 1e-5 * max(1.0, np.abs(e6).max())
    assert np.abs(f - f6).max() <= 1e-4 * scale
    assert np.abs(v - v6).max() <= 1e-5 * 400 * max(1.0, np.abs(v6).max() / 400)


@pytest.mark.parametrize("n_cfg", [1, 3, 2049])
def test_no_atoms_in_a_used_workspace(nb, n_cfg):
    """Configurations without atoms in a workspace that other work left full
    of words: the totals are zero, whatever stood where this call's chunk plan
    goes (outputs preset, so that a total that is not written shows).  The
    words, 2.0 in FP32, read as a plan whose chunks are all empty.  2,049
    configurations: the plan has a launch of its own."""
    import ctypes
    import torch
    h = I.HYPER_SMALL
    s = I.System(pos=np.zeros((0, 3)), types=np.zeros(0, np.int32), box=np.full((n_cfg, 3), 20.0),
                 atom_off=np.zeros(n_cfg + 1, np.int64))
    model = nb.Model(h, I.init_params(h).astype(np.float32))
    dsys = nb.DeviceSystem.from_inputs(s)
    nl = nb.NeighborList(0, 64, 32)
    ws = nb.Workspace(model, 0, n_cfg, 64, 32, train=True)
    words = ws.buf[:ws.buf.numel() // 4 * 4].view(torch.float32)
    out = (torch.empty(0, device="cuda"), torch.empty(3, 0, device="cuda"),
           torch.empty(n_cfg, dtype=torch.float64, device="cuda"),
           torch.empty(n_cfg, 9, dtype=torch.float64, device="cuda"))

    def fresh():
        words.fill_(2.0)
        out[2].fill_(7.0)
        out[3].fill_(7.0)

    def zero():
        assert torch.count_nonzero(out[2]).item() == 0 and torch.count_nonzero(out[3]).item() == 0

    nb.neighbors(model, dsys, nl, 0.0, ws)
    assert nb.check_list(nl) == nb.NEP_OK
    fresh()
    nb.energy_forces_virial(model, dsys, nl, ws, out=out)
    zero()
    fresh()
    nb.check(nb.lib().nep_energy_forces_virial_owned(
        model.handle, ctypes.byref(dsys.c), ctypes.byref(nl.c), 0, None, nb._ptr(out[1]), nb._ptr(out[2]),
        nb._ptr(out[3]), ws.ptr, ws.bytes, nb._stream(None)), "nep_energy_forces_virial_owned")
    zero()
    vel = torch.zeros(3, 0, device="cuda")
    for rebuild in (True, False):
        fresh()
        nb.md_step(model, dsys, nl, vel, out[1], out[2], out[3], I.MASSES.astype(np.float32), 2.0, 0.0, rebuild, ws)
        zero()
    fresh()
    zeros = torch.zeros(n_cfg, dtype=torch.float64, device="cuda")
    grad, loss = nb.param_grad(model, dsys, nl, ws, zeros, torch.zeros(3, 0, device="cuda"),
                               torch.zeros(n_cfg, 9, dtype=torch.float64, device="cuda"))
    assert torch.count_nonzero(grad).item() == 0 and loss.item() == 0.0


def test_block_sizes_stay_pinned_without_a_variant(nb):
    """A class with any launch choice but the defaults runs one thread per
    atom: block sizes chosen by set_launch also do after set_variant(-1), which
    gives up the variant only, and no longer do after set_launch()."""
    h = I.HYPER_SMALL
    s, model, dsys, nl, ws = setup(nb, h, [130, 300], 74)
    run = lambda: nb.energy_forces_virial(model, dsys, nl, ws)[1].cpu().numpy()   # noqa: E731
    default = run()
    nb.set_variant(model, 0)
    one_thread = run()
    assert not np.array_equal(default, one_thread)    # the forms' sums differ in order
    nb.set_launch(model, -1, 128, 256)
    assert np.array_equal(run(), one_thread)
    nb.set_variant(model, -1)
    assert np.array_equal(run(), one_thread)
    nb.set_launch(model, 0, 128, 0)
    nb.set_variant(model, -1)
    assert np.array_equal(run(), one_thread)
    nb.set_launch(model)
    assert np.array_equal(run(), default)
    nb.set_variant(model, 0)
    nb.set_variant(model, -1)
    assert np.array_equal(run(), default)


def test_list_build_device_box_thinner_than_the_hosts(nb):
    """The list build is chosen by the host's copy of the boxes.  Where the
    device's box of a configuration is far thinner (its rows would have more
    images than the warp build holds), the call ends with invalid input, that
    configuration's lists are empty and the others' as before."""
    h = I.HYPER_SMALL
    s, model, dsys, nl, ws = setup(nb, h, [300, 40, 200], 75)
    before = [t.cpu().numpy().reshape(-1, s.n_atoms) for t in (nl.cnt, nl.cnt_ang, nl.nbr)]
    dsys.box[1] = 0.1
    nb.neighbors(model, dsys, nl, 0.0, ws)
    assert nb.check_list(nl) == nb.NEP_ERR_INPUT
    after = [t.cpu().numpy().reshape(-1, s.n_atoms) for t in (nl.cnt, nl.cnt_ang, nl.nbr)]
    assert not after[0][:, 300:340].any() and not after[1][:, 300:340].any()
    for cols in (slice(0, 300), slice(340, 540)):
        used = np.arange(len(before[2]))[:, None] < before[0][:, cols]
        assert np.array_equal(before[0][:, cols], after[0][:, cols])
        assert np.array_equal(before[1][:, cols], after[1][:, cols])
        assert np.array_equal(before[2][:, cols][used], after[2][:, cols][used])


def wide_hidden(h, n):
    return I.Hyper(**{**h.__dict__, "n_hidden": n})


@pytest.mark.parametrize("h,total", [(I.HYPER_SMALL, 12000), (I.HYPER_SMALL, 28000), (I.HYPER_SMALL, 28001),
                                     (I.HYPER_SMALL, 38000), (I.HYPER_SMALL, 38001),
                                     (I.HYPER_TABLE2, 25000), (I.HYPER_TABLE2, 25001),
                                     (I.HYPER_TABLE2, 32000), (I.HYPER_TABLE2, 32001),
                                     (I.HYPER_LARGE, 18000), (I.HYPER_LARGE, 18001),
                                     (I.HYPER_LARGE, 27000), (I.HYPER_LARGE, 27001),
                                     (wide_hidden(I.HYPER_LARGE, 128), 10500), (wide_hidden(I.HYPER_LARGE, 128), 10501),
                                     (wide_hidden(I.HYPER_SMALL, 200), 13000), (wide_hidden(I.HYPER_SMALL, 200), 13001)],
                         ids=lambda x: str(x) if isinstance(x, int) else f"{x.dim}-{x.n_hidden}")
def test_training_forms_agree_at_the_lines(nb, h, total):
    """The loss gradient and the adjoint product on both sides of the lines
    between lane groups and one thread per atom, for models of which three,
    two and one block fit an SM, against one thread per atom; above 10,000
    atoms the lane groups' forward is the four-lane radial kernel.  Bar as in
    test_lane_groups_training_agrees_with_one_thread_per_atom."""
    import torch
    n = total // 40
    s, model, dsys, nl, _ = setup(nb, h, [n] * 39 + [total - 39 * n], 76, cap=112, cap_ang=56)
    ws = nb.Workspace(model, s.n_atoms, s.n_cfg, 112, 56, train=True)
    rng = np.random.default_rng(4)
    dev = lambda x, t: torch.tensor(np.ascontiguousarray(x), dtype=t, device="cuda")   # noqa: E731
    e = dev(rng.normal(size=s.n_cfg), torch.float64)
    f = dev(rng.normal(size=(3, s.n_atoms)), torch.float32)
    v = dev(rng.normal(size=(s.n_cfg, 9)), torch.float64)

    def grads():
        g1, loss = nb.param_grad(model, dsys, nl, ws, e, f, v)
        g2 = nb.param_grad_adjoint(model, dsys, nl, ws, e, f, v)
        return g1.cpu().numpy(), loss.item(), g2.cpu().numpy()

    got = grads()
    nb.set_variant(model, 0)
    want = grads()
    for x, y in zip(got, want):
        assert np.linalg.norm(np.asarray(x) - y) <= 1e-5 * np.linalg.norm(y)


@pytest.mark.parametrize("n,entries", [(9000, 0.5), (14000, 3.0), (21500, 3.5)])
def test_list_build_forms_agree_on_sparse_systems(nb, n, entries):
    """Gases: the line between a warp and a thread per atom falls with the
    mean list length, and with it that of the reverse search.  A configuration
    alone (below the lines) gets, entry for entry, the list of each of its two
    copies (above them); and the pairs are those of a k-d tree."""
    from scipy.spatial import cKDTree
    h = I.HYPER_SMALL
    rc = h.rc_rad
    L = np.float32((n * 4.0 / 3.0 * np.pi * rc ** 3 / entries) ** (1.0 / 3.0))
    pos = (np.random.default_rng(7).random((n, 3)) * L * 0.9999).astype(np.float32)
    types = (np.arange(n) % 3).astype(np.int32)
    model = nb.Model(h, I.init_params(h).astype(np.float32))

    def build(copies):
        s = I.System(pos=np.tile(pos, (copies, 1)), types=np.tile(types, copies),
                     box=np.full((copies, 3), L), atom_off=n * np.arange(copies + 1))
        dsys = nb.DeviceSystem.from_inputs(s)
        nl = nb.NeighborList(s.n_atoms, 64, 48)
        nb.neighbors(model, dsys, nl, 0.0, nb.Workspace(model, s.n_atoms, copies, 64, 48))
        assert nb.check_list(nl) == nb.NEP_OK, nb.last_error()
        return [t.cpu().numpy().reshape(-1, s.n_atoms) for t in (nl.cnt, nl.cnt_ang, nl.nbr, nl.rev)]

    one, two = build(1), build(2)
    used = np.arange(64)[:, None] < one[0]
    ang = np.arange(48)[:, None] < one[1]
    for c in (0, 1):
        cols = slice(c * n, (c + 1) * n)
        assert np.array_equal(one[0], two[0][:, cols]) and np.array_equal(one[1], two[1][:, cols])
        assert np.array_equal(one[2][used], two[2][:, cols][used] - c * n)
        assert np.array_equal(one[3][ang], two[3][:, cols][ang])
    # pairs nearer to the cutoff than FP32 rounds a distance in this box may go either way
    eps = 4.0 * float(L) * 2.0 ** -24
    tree = cKDTree(pos.astype(np.float64), boxsize=float(L))
    sure, maybe = (tree.query_pairs(rc + d, output_type="ndarray") for d in (-eps, eps))
    code = lambda i, j: set((np.minimum(i, j).astype(np.int64) * n + np.maximum(i, j)).tolist())   # noqa: E731
    slot, i = np.nonzero(used)
    got = code(i, one[2][slot, i])
    assert len(slot) == 2 * len(got)
    assert code(*sure.T) <= got <= code(*maybe.T)


@pytest.mark.parametrize("n,box", [(58, (3000.0, 3000.0, 3000.0)), (700, (2900.0, 500.0, 40.0)),
                                   (700, (30.0, 900.0, 3100.0)), (9000, (3050.0, 2000.0, 300.0))])
def test_list_of_atoms_in_a_nearly_empty_box(nb, n, box):
    """Boxes with far more cutoff-sized cells than twice the atoms, where the
    plan merges cells, edge by edge: the pairs are those of a k-d tree."""
    from scipy.spatial import cKDTree
    h = I.HYPER_SMALL
    box = np.array(box, np.float32)
    rng = np.random.default_rng(8)
    centre = rng.random((n // 4 + 1, 3)) * box       # small clusters, so that there are pairs
    pos = centre[rng.integers(0, len(centre), n)] + rng.normal(0.0, 3.0, (n, 3))
    pos = np.minimum((pos % box).astype(np.float32), np.nextafter(box, np.float32(0.0)))
    s = I.System(pos=pos, types=(np.arange(n) % 3).astype(np.int32), box=box[None], atom_off=np.array([0, n]))
    model = nb.Model(h, I.init_params(h).astype(np.float32))
    dsys = nb.DeviceSystem.from_inputs(s)
    nl = nb.NeighborList(n, 64, 48)
    nb.neighbors(model, dsys, nl, 0.0, nb.Workspace(model, n, 1, 64, 48))
    assert nb.check_list(nl) == nb.NEP_OK, nb.last_error()
    cnt, nbr = nl.cnt.cpu().numpy(), nl.nbr.cpu().numpy().reshape(-1, n)
    slot, i = np.nonzero(np.arange(64)[:, None] < cnt)
    code = lambda i, j: set((np.minimum(i, j).astype(np.int64) * n + np.maximum(i, j)).tolist())   # noqa: E731
    got = code(i, nbr[slot, i])
    # pairs nearer to the cutoff than FP32 rounds a distance in this box may go either way
    eps = 4.0 * float(box.max()) * 2.0 ** -24
    tree = cKDTree(pos.astype(np.float64), boxsize=box.astype(np.float64))
    sure, maybe = (tree.query_pairs(h.rc_rad + d, output_type="ndarray") for d in (-eps, eps))
    assert len(sure) > n // 2 and len(slot) == 2 * len(got)
    assert code(*sure.T) <= got <= code(*maybe.T)


def exactly(n, seed=1):
    """Rock salt with vacancies, n atoms (the last ones left out)."""
    ncell = int(np.ceil((n / 7.0) ** (1.0 / 3.0)))
    s = I.rocksalt(ncell, vacancy=0.1, seed=seed)
    assert s.n_atoms >= n
    return I.System(pos=((s.pos + 1.5) % s.box[0])[:n], types=s.types[:n], box=s.box, atom_off=np.array([0, n]))


def listed(nb, h, s, skin, precision=0):
    model = nb.Model(h, I.init_params(h, seed=5).astype(np.float32), precision=precision)
    dsys = nb.DeviceSystem.from_inputs(s)
    nl = nb.NeighborList(s.n_atoms, 160, 80)
    ws = nb.Workspace(model, s.n_atoms, s.n_cfg, 160, 80)
    nb.neighbors(model, dsys, nl, skin, ws)
    assert nb.check_list(nl) == nb.NEP_OK, nb.last_error()
    return model, dsys, nl, ws


@pytest.mark.parametrize("hname,n", [("small", 50000), ("small", 50001), ("large", 50000), ("large", 50001),
                                     ("table2", 200000), ("table2", 200001)])
def test_large_split_lines_agree_with_one_thread_per_atom(nb, hname, n):
    """The finish kernel's last lane-group size and the four-lane radial
    kernel's, and the sizes after them, on one large box."""
    s = exactly(n)
    model, dsys, nl, ws = listed(nb, MODELS[hname], s, 1.0)
    assert_close(*both_forms(nb, model, dsys, nl, ws), np.diff(s.atom_off))


@pytest.mark.parametrize("hname,precision,n", [("small", 1, 3000), ("small", 2, 3001), ("small", 1, 13500),
                                               ("small", 2, 13501), ("large", 1, 8000), ("large", 2, 8001),
                                               ("large", 1, 25000), ("large", 2, 25001)])
def test_lane_groups_16bit_network_at_the_lines(nb, hname, precision, n):
    """As test_lane_groups_16bit_network (its bars), with 32 and with 8 lanes
    per atom and with the tensor-core kernel after the four-lane radial one:
    both sides of the lines of a narrow and of a wide network."""
    s = exactly(n)
    model, dsys, nl, ws = listed(nb, MODELS[hname], s, 0.5, precision=precision)
    got, want = both_forms(nb, model, dsys, nl, ws)
    step = 2.0 ** -11 if precision == 1 else 2.0 ** -8
    assert np.abs(got[0] - want[0]).max() <= 0.5 * step
    assert np.sqrt(np.mean((got[1] - want[1]) ** 2)) <= 0.1 * step


def test_list_build_of_one_large_box(nb):
    """One box of 45,000 atoms (a warp per atom in the build and the reverse
    search) and two copies of it (a thread per atom in both): the same lists,
    entry for entry."""
    n = 45000
    s = exactly(n)
    lists = []
    for copies in (1, 2):
        batch = I.System(pos=np.tile(s.pos, (copies, 1)), types=np.tile(s.types, copies),
                         box=np.repeat(s.box, copies, 0), atom_off=n * np.arange(copies + 1))
        _, _, nl, _ = listed(nb, I.HYPER_SMALL, batch, 1.0)
        lists.append([t.cpu().numpy().reshape(-1, batch.n_atoms) for t in (nl.cnt, nl.cnt_ang, nl.nbr, nl.rev)])
    one, two = lists
    used, ang = np.arange(160)[:, None] < one[0], np.arange(80)[:, None] < one[1]
    for c in (0, 1):
        cols = slice(c * n, (c + 1) * n)
        assert np.array_equal(one[0], two[0][:, cols]) and np.array_equal(one[1], two[1][:, cols])
        assert np.array_equal(one[2][used], two[2][:, cols][used] - c * n)
        assert np.array_equal(one[3][ang], two[3][:, cols][ang])


def test_many_configurations(nb):
    """The chunk plan rides in the packing launch up to 2,048 configurations
    and has a launch of its own from there on: the totals of the same 2,048
    are the same bits, and those of E the sums of E_i."""
    h = I.HYPER_SMALL
    counts = [3, 1, 4, 2] * 512
    res = []
    for extra in ([], [5]):
        s, model, dsys, nl, ws = setup(nb, h, counts + extra, 77)
        res.append([t.cpu().numpy() for t in nb.energy_forces_virial(model, dsys, nl, ws)])
        sums = np.add.reduceat(res[-1][0].astype(np.float64), s.atom_off[:-1])
        assert np.abs(res[-1][2] - sums).max() <= 1e-12 * np.abs(sums).max()
    same = [np.array_equal(a[..., :k], b[..., :k]) for a, b, k in zip(res[0][:3], res[1][:3], (5120, 5120, 2048))]
    assert all(same) and np.array_equal(res[0][3], res[1][3][:2048])
