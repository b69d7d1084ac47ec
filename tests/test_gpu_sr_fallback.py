"""The SR step where the driver refuses the cooperative launch of the CG's vector kernel (a
context with fewer SMs than the device has): three launches make the same sums.  The refusal comes
from a fake of the call, put before a copy of the library that is linked with the shared CUDA
runtime."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = """
static int calls;
int cudaLaunchCooperativeKernel(const void* f, ...) { (void)f; ++calls; return 720; }
int fake_calls(void) { return calls; }
"""

STEPS = """
import ctypes, sys
import numpy as np, torch
from paper_1904_00031_gb300 import nk, workloads as W
lib, fake, out = sys.argv[1:4]
nk.load_library(lib)
res = {}
for k, (n, m, ns, cplx, prec) in enumerate([(40, 80, 2000, True, 1), (20, 64, 1500, False, 0),
                                            (100, 200, 3000, False, 1), (30, 90, 700, True, 0)]):
    p = W.perturb_params(W.init_params(n, m, cplx, 0.01, 3), 0.1, 4)
    r = nk.Rbm(n, m, cplx)
    r.load(p.a, p.b, p.w)
    s = torch.from_numpy(W.random_configs(ns, n, 5)).cuda()
    th = torch.empty(ns, m, dtype=r.f32_dtype(), device="cuda")
    nk.nk_rbm_theta(r, s, th)
    rng = np.random.default_rng(k)
    e = torch.from_numpy(rng.normal(size=ns) + 1j * (rng.normal(size=ns) if cplx else 0)).cuda()
    info = nk.nk_sr_step(r, s, torch.tanh(th), e, 1, 0.1, 1.0, n_cg=6, prec=prec)
    res[f"p{k}"] = np.concatenate([x.reshape(-1) for x in r.params_numpy()])
    res[f"i{k}"] = info.cpu().numpy()
res["calls"] = ctypes.CDLL(fake).fake_calls() if fake else 0
np.savez(out, **res)
"""


def test_refused_cooperative_launch(tmp_path):
    import glob

    from paper_1904_00031_gb300 import build
    build.build()
    fake, lib = str(tmp_path / "libfake.so"), str(tmp_path / "libnk_shared.so")
    (tmp_path / "fake.c").write_text(FAKE)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", fake, str(tmp_path / "fake.c")], check=True)
    subprocess.run([build.nvcc(), "-shared", "-cudart", "shared"] + build.ARCH + ["-o", lib] +
                   sorted(glob.glob(os.path.join(build.BUILD, "*.o"))), check=True)
    out = {}
    for name, pre in (("fused", ""), ("refused", fake)):
        f = str(tmp_path / (name + ".npz"))
        env = dict(os.environ, PYTHONPATH=ROOT)
        if pre:
            env["LD_PRELOAD"] = pre
        run = subprocess.run([sys.executable, "-c", STEPS, lib, pre, f], cwd=ROOT, env=env,
                             capture_output=True, text=True, timeout=300)
        assert run.returncode == 0, run.stderr[-2000:]
        out[name] = np.load(f)
    assert out["refused"]["calls"] == 4  # one refusal a step
    for k in range(4):
        for x in ("p", "i"):
            assert np.isfinite(out["fused"][f"{x}{k}"]).all()
            assert np.array_equal(out["fused"][f"{x}{k}"], out["refused"][f"{x}{k}"]), (x, k)
