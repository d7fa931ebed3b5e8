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
