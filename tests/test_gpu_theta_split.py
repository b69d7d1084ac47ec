"""FP32 theta and tanh(theta) whose hidden tiles are dealt to several CTAs (few samples): bit for
bit those of a large call, which runs one CTA per 64 samples, alone and in a batch; the backward,
which takes tanh(theta) the same way, against the FP64 oracle."""
import numpy as np
import pytest
import torch

from oracle import rbm as orbm
from paper_1904_00031_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nk():
    from paper_1904_00031_gb300 import build, nk as nkmod
    build.build()
    nkmod.load_library()
    return nkmod


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("n,m", [(9, 1), (40, 64), (40, 65), (33, 200), (100, 700)])
def test_theta_of_few_samples(nk, n, m, cplx):
    p = W.perturb_params(W.init_params(n, m, cplx, 0.01, m), 0.1, 8)
    r = nk.Rbm(n, m, cplx)
    r.load(p.a, p.b, p.w)
    s = torch.from_numpy(W.random_configs(20000, n, 3)).cuda()
    big = torch.empty(20000, m, dtype=r.f32_dtype(), device="cuda")
    nk.nk_rbm_theta(r, s, big)
    jobs = []
    for ns in (1, 63, 300, 6001):
        th = torch.full((ns, m), float("nan"), dtype=r.f32_dtype(), device="cuda")
        nk.nk_rbm_theta(r, s[:ns].contiguous(), th)
        assert torch.equal(th, big[:ns]), ns
        jobs.append(dict(rbm=r, sigma=s[:ns].contiguous(), logpsi_out=None,
                         theta_out=torch.full_like(th, float("nan"))))
    for k in (2, 4):
        nk.nk_batch_logpsi(jobs[:k])
        for j in jobs[:k]:
            assert torch.equal(j["theta_out"], big[:len(j["sigma"])])
    ns = 300
    g = np.random.default_rng(1).normal(size=ns) / ns
    got = nk.nk_rbm_logpsi_backward(r, s[:ns].contiguous(), torch.from_numpy(g + 0j).cuda())
    sig, t = orbm.logderiv_factored(p, s[:ns].cpu().numpy())
    ref = np.concatenate([(g[:, None] * sig).sum(0), (g[:, None] * t.conj()).sum(0),
                          ((g[:, None] * t.conj()).T @ sig).reshape(-1)])
    assert np.linalg.norm(got.cpu().numpy() - ref) <= 1e-4 * np.linalg.norm(ref)
