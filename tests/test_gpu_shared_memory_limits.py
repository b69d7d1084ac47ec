"""Calls from several host threads on streams of their own: a kernel's limit on dynamic shared
memory is one per function, so a call that needs little must not take it from one that needs
much."""
import threading

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


def run_threads(calls, reps):
    """Every call in a thread of its own, reps times; the exceptions they raised."""
    errors, start = [], threading.Barrier(len(calls))

    def work(fn):
        st = torch.cuda.Stream()
        torch.zeros(1, device="cuda")  # binds the thread to the device
        start.wait()
        try:
            for _ in range(reps):
                fn(st)
            st.synchronize()
        except Exception as e:  # noqa: BLE001 (reported by the caller)
            errors.append(e)

    ts = [threading.Thread(target=work, args=(fn,)) for fn in calls]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    return errors


def energy_call(nk, op, n, m, cplx, ns):
    p = W.perturb_params(W.init_params(n, m, cplx, 0.01, 5), 0.1, 9)
    r = nk.Rbm(n, m, cplx)
    r.load(p.a, p.b, p.w)
    s = torch.from_numpy(W.random_configs(ns, n, 2, cplx)).cuda()
    th = torch.empty(ns, m, dtype=r.f32_dtype(), device="cuda")
    nk.nk_rbm_logpsi(r, s, theta_out=th)
    gop = nk.Operator(op)
    e = torch.empty(ns, dtype=torch.complex128, device="cuda")
    sc = nk.local_energy_scratch(r, gop)
    fn = lambda st: nk.nk_local_energy(r, gop, s, th, e, scratch=sc, stream=st)
    fn(None)
    torch.cuda.synchronize()
    return fn, e, e.clone()


def sr_call(nk, n, m, ns):
    p = W.perturb_params(W.init_params(n, m, False, 0.01, 3), 0.1, 4)
    r = nk.Rbm(n, m, False)
    r.load(p.a, p.b, p.w)
    s = torch.from_numpy(W.random_configs(ns, n, 5)).cuda()
    t = torch.rand(ns, m, device="cuda")
    e = torch.randn(ns, dtype=torch.float64, device="cuda").to(torch.complex128)
    sc = nk.sr_scratch(r, ns)
    info = torch.zeros(nk.NK_INFO_LEN, dtype=torch.float64, device="cuda")
    fn = lambda st: nk.nk_sr_step(r, s, t, e, 1, 0.1, 0.0, 3, 1e-12, scratch=sc, info_out=info,
                                  stream=st)
    fn(None)
    torch.cuda.synchronize()
    return fn, info, info.clone()


def sweep_call(nk, n, m, nc):
    p = W.init_params(n, m, False, 0.01, 3)
    r = nk.Rbm(n, m, False)
    r.load(p.a, p.b, p.w)
    ch = nk.Chains(W.init_chains(nc, n, False, 8), 8, 7)
    sc = nk.metropolis_scratch(r, nk.NK_MOVE_FLIP, n)
    s = torch.empty(nc, n, dtype=torch.int8, device="cuda")
    fn = lambda st: nk.nk_metropolis_sweep(r, ch, nk.NK_MOVE_FLIP, None, None, 0, 1,
                                           samples_out=s, scratch=sc, stream=st)
    fn(None)
    torch.cuda.synchronize()
    return fn, None, None


def logpsi_call(nk, n, m):
    p = W.perturb_params(W.init_params(n, m, True, 0.01, 5), 0.1, 9)
    r = nk.Rbm(n, m, True)
    r.load(p.a, p.b, p.w)
    s = torch.from_numpy(W.random_configs(200, n, 2)).cuda()
    lp = torch.empty(200, dtype=torch.complex128, device="cuda")
    fn = lambda st: nk.nk_rbm_logpsi(r, s, prec=nk.NK_PREC_BF16X2, logpsi_out=lp, stream=st)
    fn(None)
    torch.cuda.synchronize()
    return fn, lp, lp.clone()


@pytest.mark.parametrize("what", ["energies", "sr", "sweeps", "logpsi"])
def test_calls_of_different_sizes_in_threads(nk, what):
    if what == "energies":  # clusters, CTAs alone on their SMs or not
        op = W.ising(289, W.square_bonds(17), h=3.04)
        calls = [energy_call(nk, op, 289, 35, False, ns) for ns in (300, 1500, 2500, 4000, 5000, 8000)]
    elif what == "sr":      # the whole CG in one cluster, shared memory by the sample count
        calls = [sr_call(nk, 10, 10, ns) for ns in (100, 600, 2000, 3900)]
    elif what == "sweeps":
        calls = [sweep_call(nk, n, 64, 64) for n in (10, 80)]
    else:
        calls = [logpsi_call(nk, n, 40) for n in (9, 400)]
    assert run_threads([c[0] for c in calls], 4000) == []
    for _, out, ref in calls:
        if out is not None:
            assert torch.equal(torch.view_as_real(out) if out.is_complex() else out,
                               torch.view_as_real(ref) if ref.is_complex() else ref)
