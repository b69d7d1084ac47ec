"""a . sigma in the tensor-core ln psi: with W = b = 0 ln psi is a . sigma plus the same ln cosh 0
for every unit, which a second RBM with a = 0 gives."""
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


def visible(nk, a, s, m=70):
    """ln psi minus its hidden part, and the hidden part's size."""
    n, cplx = len(a), np.iscomplexobj(a)
    out = []
    for aa in (a, np.zeros_like(a)):
        r = nk.Rbm(n, m, cplx)
        r.load(aa, np.zeros(m, a.dtype), np.zeros((m, n), a.dtype))
        out.append(nk.nk_rbm_logpsi(r, torch.from_numpy(s).cuda(), prec=nk.NK_PREC_BF16X2)
                   .cpu().numpy())
    return out[0] - out[1], np.abs(out[1]).max()


def exact(a, s):
    """a . sigma in extended precision, as a pair (re, im) of long doubles."""
    part = lambda x: (s.astype(np.longdouble) * x.astype(np.longdouble)).sum(1)
    return part(a.real), part(a.imag) if np.iscomplexobj(a) else np.zeros(len(s), np.longdouble)


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("n,ns,scale", [(1, 3, 1.0), (7, 129, 1.0), (8, 64, 1e-200),
                                        (130, 300, 1.0), (400, 300, 1.0), (447, 300, 1e3)])
def test_visible_term_to_64_bits(nk, n, ns, scale, cplx):
    """As accurate as a plain FP64 sum is on average: each of the n addends within half a unit
    in the last place of the largest |a_i|, and three roundings of the result (the sum's, and
    of the two additions of the hidden part)."""
    rng = np.random.default_rng(n)
    a = rng.normal(size=n) * scale
    if cplx:
        a = a + 1j * rng.normal(size=n) * scale
    s = W.random_configs(ns, n, 3)
    v, hidden = visible(nk, a, s)
    for got, ref, ai in ((v.real, exact(a, s)[0], a.real), (v.imag, exact(a, s)[1], a.imag)):
        tol = n * 2.0 ** -53 * np.abs(ai).max() + 3 * 2.0 ** -53 * (np.abs(ref) + hidden)
        assert np.all(np.abs(got - ref) <= tol), (np.abs(got - ref) / tol).max()


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("big", [1e39, -3e300, np.inf])
def test_visible_bias_beyond_float(nk, big, cplx):
    n, ns = 21, 150
    a = np.random.default_rng(2).normal(size=n).astype(complex if cplx else float)
    a[5] = big
    s = W.random_configs(ns, n, 4)
    v, _ = visible(nk, a, s)
    if np.isinf(big):
        assert np.array_equal(v.real, big * s[:, 5])
    else:
        ref = exact(a, s)[0]
        assert np.all(np.abs(v.real - ref) <= 1e-15 * np.abs(ref))
    # the other part is what it would be without the large bias
    ref = exact(a, s)[1]
    assert np.all(np.abs(v.imag - ref) <= n * 2.0 ** -53 * 4 + 4e-16 * np.abs(ref))
