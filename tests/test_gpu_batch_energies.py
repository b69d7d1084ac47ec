"""nk_batch_local_energy over problems of every form (one or more move tiles, whole ones, site
quads, no moves; a cluster, one CTA or a shared range of CTAs per configuration tile): bit for bit
the single calls, in launches that the problems share."""
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


def operator(which, n):
    if which == "tfim":
        return W.ising(n, W.chain_bonds(n), h=1.0)
    if which == "classical":  # no moves
        return W.ising(n, W.chain_bonds(n), h=0.0)
    if which == "heis":
        return W.heisenberg(n, W.chain_bonds(n), 1.0, True, W.sublattice(n))
    return W.j1j2(8, 1.0, 0.5, True)


def job(nk, which, n, cplx, ns, m):
    p = W.perturb_params(W.init_params(n, m, cplx, 0.01, n + m), 0.3 / np.sqrt(n), ns)
    r = nk.Rbm(n, m, cplx)
    r.load(p.a, p.b, p.w)
    s = torch.from_numpy(W.random_configs(ns, n, 21 + n, which not in ("tfim", "classical"))).cuda()
    th = torch.empty(ns, m, dtype=r.f32_dtype(), device="cuda")
    nk.nk_rbm_theta(r, s, th)
    op = nk.Operator(operator(which, n))
    return dict(rbm=r, op=op, sigma=s, theta=th, t_out=torch.zeros_like(th),
                eloc_out=torch.full((ns,), float("nan"), dtype=torch.complex128, device="cuda"),
                scratch=nk.local_energy_scratch(r, op))


MIX = [("tfim", 289, False, 300, 35), ("tfim", 289, False, 6000, 35), ("tfim", 289, False, 39001, 5),
       ("tfim", 100, False, 77, 40), ("tfim", 64, False, 1000, 33), ("tfim", 20, False, 5, 65),
       ("classical", 20, False, 100, 12), ("tfim", 70, True, 300, 20), ("heis", 64, True, 300, 64),
       ("heis", 64, True, 5000, 17), ("heis", 128, True, 1000, 20), ("heis", 30, True, 129, 40),
       ("classical", 20, True, 100, 12), ("j1j2", 64, True, 300, 33), ("j1j2", 64, True, 6000, 33),
       ("j1j2", 64, True, 39001, 9), ("j1j2", 64, False, 700, 33)]


@pytest.mark.parametrize("pick", [slice(None), slice(0, 3), slice(8, 10), slice(13, 14),
                                  slice(3, 7)], ids=str)
def test_batch_equals_single_calls(nk, pick):
    jobs = [job(nk, *c) for c in MIX[pick]]
    ref = []
    for j in jobs:
        t = torch.zeros_like(j["t_out"])
        ref.append((nk.nk_local_energy(j["rbm"], j["op"], j["sigma"], j["theta"], t_out=t), t))
    nk.nk_batch_local_energy(jobs)
    for c, j, (e, t) in zip(MIX[pick], jobs, ref):
        assert torch.isfinite(torch.view_as_real(e)).all(), c
        assert torch.equal(j["eloc_out"], e) and torch.equal(j["t_out"], t), c


@pytest.mark.parametrize("which,cplx,n", [("tfim", False, 80), ("heis", True, 64),
                                          ("j1j2", True, 64)])
def test_problems_share_launches(nk, which, cplx, n):
    """Seventy problems of one shape: the move tables and at most both forms of the energy
    kernel, each in two launches of up to 64 problems."""
    jobs = [job(nk, which, n, cplx, 64, 16)] * 70
    nk.nk_batch_local_energy(jobs)
    assert nk.count_kernels(lambda: nk.nk_batch_local_energy(jobs)) <= (6 if cplx else 4)
