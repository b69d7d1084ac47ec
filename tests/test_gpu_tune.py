"""nk_tune_shapes on real RBMs and site-quad operators, whose local energies run the same split
whatever eloc_segs says: a tuned call gives the bits of an untuned one, every time.  (The count
orders a product's factors, so one that was chosen by timing would not.)"""
import numpy as np
import pytest
import torch

from paper_1904_00031_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nk():
    from paper_1904_00031_gb300 import build, nk as nkmod
    build.build()
    nkmod.load_library()
    return nkmod


def bonds_of_four(n):
    """Four bonds per site of a ring: whole move tiles in site quads."""
    i = np.arange(n)
    return np.concatenate([np.stack([i, (i + d) % n], 1) for d in (1, 2, 3, 4)])


# (two and three move tiles: the counts order the second tile's factors differently)
@pytest.mark.parametrize("which,cplx", [("tfim", False), ("quads", True), ("heis", True)])
@pytest.mark.parametrize("ns", [300, 3000, 20000])
def test_tuned_energies(nk, which, cplx, ns):
    n, op = {"tfim": (100, W.ising(100, W.square_bonds(10), h=3.04)),
             "quads": (48, W.heisenberg(48, bonds_of_four(48), 1.0, False, W.sublattice(48))),
             "heis": (130, W.heisenberg(130, W.chain_bonds(130), 1.0, True, W.sublattice(130)))}[which]
    m = 100
    p = W.perturb_params(W.init_params(n, m, cplx, 0.01, 5), 0.3 / np.sqrt(n), 9)
    r = nk.Rbm(n, m, cplx)
    r.load(p.a, p.b, p.w)
    s = torch.from_numpy(W.random_configs(ns, n, 21, which != "tfim")).cuda()
    th = torch.empty(ns, m, dtype=r.f32_dtype(), device="cuda")
    nk.nk_rbm_theta(r, s, th)
    gop = nk.Operator(op)
    sc = nk.local_energy_scratch(r, gop)
    ref = nk.nk_local_energy(r, gop, s, th, scratch=sc)
    for _ in range(12):
        tmp, e = torch.empty_like(th), torch.empty_like(ref)
        _, segs = nk.nk_tune_shapes(r, gop, s, tmp, e, sc)
        assert segs in (1, 2)
        nk.nk_local_energy(r, gop, s, th, eloc_out=e, scratch=sc)
        if which != "heis":  # (a split that is timed: the same to the sums' rounding)
            assert torch.equal(e, ref)
        assert (e - ref).abs().max() <= 1e-12 * ref.abs().max()
