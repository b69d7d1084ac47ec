"""nk_sr_step in FP32 where the whole conjugate gradient runs in one cluster (few parameters and
samples) and just beyond, against the FP64 oracle: one to four steps of 16 columns, a ragged last
tile of 64 samples, CTAs without a tile, one and several sample splits, rows of even and odd
pitch, weights, both fields; and convergence before the last iteration.  The direction after a
fixed number of CG iterations within 1e-3, as in the per-entry parity tests."""
import numpy as np
import pytest
import torch

from oracle import rbm as orbm
from oracle import sr as osr
from paper_1904_00031_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nk():
    from paper_1904_00031_gb300 import build, nk as nkmod
    build.build()
    nkmod.load_library()
    return nkmod


def inputs(n, m, ns, cplx, weighted):
    p = W.perturb_params(W.init_params(n, m, cplx, 0.01, 3), 0.3 / np.sqrt(n), 4)
    s = W.random_configs(ns, n, 5)
    rng = np.random.default_rng(6)
    e = rng.normal(size=ns) + 1j * (rng.normal(size=ns) if cplx else 0.0)
    w = rng.uniform(0.5, 1.5, ns) if weighted else None
    if weighted:
        w /= w.sum()
    return p, s, e, w


def step(nk, p, s, e, w, t32, shift, its, rtol):
    """(FP64 direction of the update, info) of one step with learning rate 1."""
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    r = nk.Rbm(p.n, p.m, p.is_complex)
    r.load(p.a, p.b, p.w)
    info = nk.nk_sr_step(r, dev(s), dev(t32), dev(e), 1, shift, 1.0, n_cg=its, cg_rtol=rtol,
                         weights=None if w is None else dev(w))
    a, b, ww = r.params_numpy()
    return p.flat() - np.concatenate([a, b, ww.reshape(-1)]), nk.info_dict(info)


CASES = [(14, 14, 1500, True, True), (15, 63, 600, False, True), (7, 17, 513, True, False),
         (10, 10, 1008, False, False), (15, 30, 1001, True, False), (31, 31, 511, False, True),
         (20, 40, 600, True, True), (3, 47, 65, False, False), (1, 1, 64, True, False),
         (10, 10, 2100, False, True),
         # beyond the rule: a second round of the adjoint, more tiles, 1025 parameters, 64 units
         (15, 63, 1000, True, True), (20, 20, 1500, False, False), (8, 8, 4000, True, False),
         (40, 24, 600, False, True), (9, 64, 600, True, False)]


@pytest.mark.parametrize("n,m,ns,cplx,weighted", CASES)
def test_direction(nk, n, m, ns, cplx, weighted):
    p, s, e, w = inputs(n, m, ns, cplx, weighted)
    sig, t = orbm.logderiv_factored(p, s)
    t32 = t.astype(np.complex64 if cplx else np.float32)
    f = osr.force_lazy(sig, t32, e, n, m, w, not cplx)
    its = 4
    x, _, _ = osr.cg(lambda v: osr.sr_matvec_lazy(sig, t32.astype(t.dtype), v, n, m, w, not cplx),
                     f, 0.1, its, 1e-12)
    d, info = step(nk, p, s, e, w, t32, 0.1, its, 1e-12)
    assert info["cg_iters"] == min(its, n + m + n * m)  # (exact in as many as there are parameters)
    assert abs(info["f_norm"] - np.linalg.norm(f)) <= 1e-5 * np.linalg.norm(f)
    assert np.linalg.norm(d - x) <= 1e-3 * np.linalg.norm(x)


@pytest.mark.parametrize("n,m,ns,cplx,weighted", CASES[:6])
def test_convergence(nk, n, m, ns, cplx, weighted):
    """Converged early: the solution of the dense system, to the residual that was asked for
    (1e-4; with a shift of 1 the system's condition number is that of S + 1, below 1e3)."""
    p, s, e, w = inputs(n, m, ns, cplx, weighted)
    _, t = orbm.logderiv_factored(p, s)
    t32 = t.astype(np.complex64 if cplx else np.float32)
    d, info = step(nk, p, s, e, w, t32, 1.0, 500, 1e-4)
    assert 1 < info["cg_iters"] < 500 and info["cg_resid"] <= 1e-4 and info["flags"] == 0
    sig = s.astype(np.float64)
    f = osr.force_lazy(sig, t32, e, n, m, w, not cplx)
    r = osr.sr_matvec_lazy(sig, t32.astype(t.dtype), d, n, m, w, not cplx) + d - f
    # the residual asked for, and the FP32 contractions' error in S d (1e-6 of it a piece)
    assert np.linalg.norm(r) <= 1e-4 * np.linalg.norm(f) + 1e-5 * np.linalg.norm(f - d)
