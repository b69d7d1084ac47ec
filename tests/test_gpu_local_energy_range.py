"""Local energies whose running products leave FP32's range: large factors for the first
hidden units, small ones for the rest, so that the ratio itself is ordinary.  Only site 0 is
coupled (W[:, i > 0] = 0), so every move that flips it has the same ratio and all the others 1;
theta is given, which makes a unit's factor cosh c - s tanh(theta) sinh c as wanted."""
import itertools

import numpy as np
import pytest
import torch

from oracle import local_energy as ole
from paper_1904_00031_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nk():
    from paper_1904_00031_gb300 import build, nk as nkmod
    build.build()
    nkmod.load_library()
    return nkmod


def operator(which):
    if which == "ising":
        return W.ising(2, np.array([[0, 1]]), h=1.0)
    if which == "quads":  # complex RBMs: the site-quad layout
        return W.j1j2(8, 1.0, 0.5, True)
    return W.heisenberg(70, W.chain_bonds(70), 1.0, True, W.sublattice(70))


def energy_parts(op, s):
    """(E of everything that leaves site 0 alone, sum of the elements that flip it) of the
    configuration s: E_loc = first + second * ratio."""
    rest = flip = 0.0
    for sites, mat in ole._outcomes(op):
        row = 0
        for i in sites:
            row = 2 * row + (1 - int(s[i])) // 2
        for o in itertools.product((0, 1), repeat=len(sites)):
            col = int("".join(map(str, o)), 2)
            mel = mat[row, col]
            if any(i == 0 and 1 - 2 * x != s[i] for i, x in zip(sites, o)):
                flip += mel
            else:
                rest += mel
    return rest, flip


def energies(nk, which, w0, theta, configs):
    """(local energies, their parts) with W[:, 0] = w0 and the given theta [m]."""
    op = operator(which)
    cplx = which != "ising"
    n, m = op.n, len(w0)
    w = np.zeros((m, n), dtype=complex if cplx else float)
    w[:, 0] = w0
    r = nk.Rbm(n, m, cplx)
    r.load(np.zeros(n, w.dtype), np.zeros(m, w.dtype), w)
    th = torch.as_tensor(np.tile(theta, (len(configs), 1))).to(r.f32_dtype()).cuda()
    e = nk.nk_local_energy(r, nk.Operator(op), torch.from_numpy(configs).cuda(), th)
    return e.cpu().numpy(), [energy_parts(op, s) for s in configs]


def neel(which, up):
    n = operator(which).n
    x = np.arange(n)
    if which == "quads":
        x = x % 8 + x // 8
    s = np.where(x % 2 == 0, 1, -1).astype(np.int8)
    return s if up else -s


@pytest.mark.parametrize("which", ["ising", "quads", "chain"])
def test_product_just_below_the_largest_float(nk, which):
    """The product between two renormalisations (8 real or 16 complex units) in [2^127, 2^128):
    finite, and has to stay what it is.  (A move tile that takes the units in the other
    direction comes to them with a mantissa of 2^0.74: 2^127.84.)"""
    k = 8 if which == "ising" else 16
    up = np.arccosh(2.0 ** (127.1 / k)) / 2
    # then 112 units of exp(-0.8): cosh c - sinh c loses (C + S) / (C - S) = 5 roundings of 6e-8
    # a unit, 3.4e-5 in all at worst
    w0 = np.concatenate([np.full(k, up), np.full(112, 0.4)])
    theta = np.concatenate([np.zeros(k), np.full(112, 20.0)])
    e, parts = energies(nk, which, w0, theta, neel(which, True)[None])
    ratio = np.cosh(2 * up) ** k * np.exp(-0.8 * 112)
    ref = parts[0][0] + parts[0][1] * ratio
    assert 0.1 < ratio < 1 and abs(e[0] - ref) <= 1e-4 * abs(ref)


def test_infinite_product_keeps_its_sign(nk):
    """A product of positive factors that overflows in the second group of 8 units of 32 is
    renormalised three times afterwards."""
    w0 = np.concatenate([np.zeros(8), np.full(4, 14.0)])
    e, parts = energies(nk, "ising", w0, np.zeros(12), np.array([[1, -1]], dtype=np.int8))
    assert parts[0][1].real < 0 and e[0].real < -1e40


def theta_of_one(nk, cplx):
    """A theta with tanh(+-theta) = +-1 to the bit."""
    grid = np.arange(10.0, 20.0, 0.25)
    r = nk.Rbm(1, len(grid), cplx)
    z = torch.as_tensor(np.stack([grid, -grid])).to(r.f32_dtype()).cuda()
    t = nk.nk_logderiv(r, torch.ones(2, 1, dtype=torch.int8, device="cuda"), z).cpu().numpy()
    return grid[np.nonzero((t[0] == 1) & (t[1] == -1))[0][0]]


# Exponents that go far beyond 16 bits and come back: cosh c +- sinh c with c = k ln 2 is
# exactly 2^(+-k), and cosh c and sinh c are exact in FP32 for k <= 11, so the ratio is exactly
# 1.  The two configurations of a pair go in opposite directions.  Exponents are packed into 16
# bits each up to 2040 real or 4080 complex units and kept apart beyond: either side of the
# line, and a count that reaches 33,000 (28,000 in complex RBMs, of 8192 units at most).
@pytest.mark.parametrize("which,m", [("ising", 800), ("ising", 2040), ("ising", 2041),
                                     ("ising", 6016), ("quads", 1600), ("quads", 4080),
                                     ("quads", 4081), ("quads", 8192)])
def test_exponents_out_and_back(nk, which, m):
    k = 11 if which == "ising" else 7
    n = operator(which).n
    half, one = m // 2, theta_of_one(nk, which != "ising")
    theta = np.zeros(m)
    theta[:half], theta[half:2 * half] = -one, one
    w0 = np.full(m, k * np.log(2.0) / 2)
    w0[2 * half:] = 0.0
    s = np.stack([neel(which, up) for up in (True, False, True)])
    e, parts = energies(nk, which, w0, theta, s)
    for x, (rest, flip) in zip(e, parts):
        # sums of up to 200 elements of order 1 in FP64
        assert abs(x - (rest + flip)) <= 1e-12 * (abs(rest) + abs(flip) + n), (x, rest, flip)


@pytest.mark.parametrize("which,m", [("ising", 2040), ("ising", 8192), ("quads", 4080),
                                     ("quads", 8192)])
def test_exponents_to_the_end(nk, which, m):
    """All units one way: 2^(+-22,440) to 2^(+-90,112), infinite in one configuration of a pair
    and nothing in the other."""
    k = 11 if which == "ising" else 7
    w0 = np.full(m, k * np.log(2.0) / 2)
    s = np.stack([neel(which, up) for up in (True, False)])
    assert s[0, 0] == 1
    e, parts = energies(nk, which, w0, np.full(m, -theta_of_one(nk, which != "ising")), s)
    assert parts[0][1].real < 0 and e[0].real == -np.inf
    assert abs(e[1] - parts[1][0]) <= 1e-12 * (abs(parts[1][0]) + s.shape[1])
