"""Sweeps on either side of the sampler's rules on the number of CTAs (128 or 64 registers per
thread; rows resident or through the ring): the first chains of a launch of any size follow the
oracle's trajectories, bit for bit where no decision came within 1e-3 of a tie."""
import numpy as np
import pytest
import torch

from oracle import sampler as osam
from paper_1904_00031_gb300 import workloads as W

pytestmark = pytest.mark.gpu
SEED, COUNTER = 0xBADC0DE, 96


@pytest.fixture(scope="module")
def nk():
    from paper_1904_00031_gb300 import build, nk as nkmod
    build.build()
    nkmod.load_library()
    return nkmod


def problem(nk, move, n, m, cplx, G, nc):
    """(sweep arguments, oracle trajectories of the first 5 groups, their margins)."""
    p = W.perturb_params(W.init_params(n, m, cplx, 0.01, 7 + m), 0.5 / np.sqrt(n), 3)
    s0 = W.init_chains(nc, n, move == "exchange", 8)
    bonds = W.chain_bonds(n).astype(np.int32)
    k = 5 * G
    ref = osam.metropolis(p, s0[:k], move, bonds, G, SEED, COUNTER, 1, 1, return_margin=True)
    r = nk.Rbm(n, m, cplx)
    r.load(p.a, p.b, p.w)
    r._s.sampler = 1
    ch = nk.Chains(s0, G, SEED)
    ch.counter = COUNTER
    mv = nk.NK_MOVE_FLIP if move == "flip" else nk.NK_MOVE_EXCHANGE
    b = torch.from_numpy(bonds).cuda()
    job = dict(rbm=r, chains=ch, move=mv, bond_i=b[:, 0].contiguous(),
               bond_k=b[:, 1].contiguous(), n_discard=1, n_samples_per_chain=1,
               samples_out=torch.zeros(nc, n, dtype=torch.int8, device="cuda"),
               n_accept_out=torch.zeros(nc, dtype=torch.int64, device="cuda"),
               scratch=nk.metropolis_scratch(r, mv, n))
    return job, ref[0].reshape(k, n), ref[3], ref[4]


def check(job, samp, nacc, marg):
    ok = marg > 1e-3
    k = len(ok)
    assert ok.sum() >= k // 4
    assert np.array_equal(job["samples_out"].cpu().numpy()[:k][ok], samp[ok])
    assert np.array_equal(job["n_accept_out"].cpu().numpy()[:k][ok], nacc[ok])


# threads per CTA: 32 G, twice that from 512 units on; at 128 registers 512 threads fit an SM
@pytest.mark.parametrize("move,n,m,cplx,G", [
    ("flip", 24, 128, False, 8), ("flip", 24, 200, False, 4), ("flip", 24, 400, False, 8),
    ("flip", 24, 512, False, 8), ("flip", 24, 700, False, 8), ("flip", 24, 1000, False, 8),
    ("exchange", 16, 64, True, 8), ("exchange", 16, 128, True, 4)])
@pytest.mark.parametrize("over", [0, 1])
def test_registers_per_thread(nk, move, n, m, cplx, G, over):
    line = 152 * (512 // (32 * G * (2 if m >= 512 else 1)))
    job, *ref = problem(nk, move, n, m, cplx, G, (line + over) * G)
    nk.nk_metropolis_sweep(**job)
    check(job, *ref)


@pytest.mark.parametrize("chains", [(64, 1240, 1232), (1232, 1240, 64, 80)])
def test_batch_registers_per_thread(nk, chains):
    """Below 305 CTAs of a template in all, and above."""
    probs = [problem(nk, "flip", 24, 100 + u, False, 8, nc) for u, nc in enumerate(chains)]
    nk.nk_batch_sweep([j for j, *_ in probs])
    for j, *ref in probs:
        check(j, *ref)


# The rows' bytes leave room for three CTAs per SM (of eight by registers), one (of four), two,
# three (which is enough beyond what fits at once, too).
@pytest.mark.parametrize("move,n,m,cplx,G,fit", [("flip", 24, 256, False, 4, 3),
                                                 ("flip", 96, 192, False, 8, 1),
                                                 ("exchange", 130, 32, True, 8, 2),
                                                 ("flip", 24, 256, False, 8, 3)])
@pytest.mark.parametrize("over", [0, 1])
def test_batch_rows(nk, move, n, m, cplx, G, fit, over):
    """As many CTAs in a call as fit with their rows resident, and one more."""
    ctas = 152 * fit + over
    probs = [problem(nk, move, n, m, cplx, G, k * G) for k in (40, ctas - 90, 50)]
    nk.nk_batch_sweep([j for j, *_ in probs])
    for j, *ref in probs:
        check(j, *ref)
