"""The launch counts that an iteration reports against the kernel nodes of its captured graph,
on either side of the library's dispatch rules."""
import ctypes

import pytest
import torch

from paper_1904_00031_gb300 import workloads as W

pytestmark = pytest.mark.gpu

FP32, BF16X2 = 0, 1


@pytest.fixture(scope="module")
def nk():
    from paper_1904_00031_gb300 import build, nk as nkmod
    build.build()
    nkmod.load_library()
    return nkmod


def kernels(fn):
    """Kernel nodes of fn() captured into a graph (which is not run)."""
    fn()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        fn()
    cu = ctypes.CDLL("libcuda.so.1")
    graph, cnt = ctypes.c_void_p(g.raw_cuda_graph()), ctypes.c_size_t(0)
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(cnt)) == 0
    nodes = (ctypes.c_void_p * cnt.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(cnt)) == 0
    total, kind = 0, ctypes.c_int(0)
    for node in nodes:
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        total += kind.value == 0  # CU_GRAPH_NODE_TYPE_KERNEL
    return total


def tfim(n, m, chains, per=1, cg=3):
    return W.Workload("tfim", n, m, False, W.ising(n, W.chain_bonds(n), h=1.0), "flip",
                      W.chain_bonds(n), False, chains, per, 1, 0.01, 0.01, cg, 5)


def heis(n, m, chains, per=1, cg=3):
    return W.Workload("heis", n, m, True,
                      W.heisenberg(n, W.chain_bonds(n), 1.0, True, W.sublattice(n)), "exchange",
                      W.chain_bonds(n), True, chains, per, 1, 0.01, 0.01, cg, 5)


def j1j2(L, chains, cg=3):
    n = L * L
    return W.Workload("j1j2", n, n, True, W.j1j2(L, 1.0, 0.5, True), "exchange",
                      W.square_bonds(L), True, chains, 1, 1, 0.01, 0.01, cg, 5, lattice="square")


# FP32: either side of the one-cluster CG's lines (1024 parameters, 63 units, 4096 samples, the
# products by field), the adjoint with and without its own centring, more centring partials than
# fit; BF16 hi + lo: centring by the adjoint, by a launch, by two; site quads, whole move tiles.
@pytest.mark.parametrize("w,prec", [
    (tfim(10, 10, 16, 63), FP32), (tfim(10, 10, 4104), FP32), (tfim(20, 40, 1216), FP32),
    (tfim(20, 40, 1224), FP32), (tfim(20, 20, 1544), FP32), (tfim(10, 64, 512), FP32),
    (tfim(31, 31, 512), FP32), (tfim(32, 31, 512), FP32), (tfim(100, 400, 2048), FP32),
    (tfim(8, 8, 131200), FP32), (heis(14, 14, 1496), FP32), (heis(20, 40, 400), FP32),
    (heis(20, 40, 1000), FP32), (heis(14, 14, 1160), FP32), (heis(14, 14, 3000), FP32),
    (heis(64, 64, 512), FP32), (tfim(40, 80, 512), BF16X2), (heis(64, 64, 512), BF16X2),
    (heis(64, 256, 512), BF16X2), (heis(62, 256, 65536), BF16X2), (j1j2(8, 256), BF16X2),
    (j1j2(8, 256), FP32)], ids=lambda x: getattr(x, "name", x))
def test_iteration(nk, w, prec):
    from paper_1904_00031_gb300.vmc import VmcSr
    v = VmcSr(w, W.init_params(w.n, w.m, w.is_complex, 0.01, 3), prec=prec, graph=True)
    assert kernels(v._eager_step) == v.launches_per_step()


@pytest.mark.parametrize("prec", [FP32, BF16X2])
def test_symmetric_iteration(nk, prec):
    from paper_1904_00031_gb300.vmc import VmcSrSymm
    w = tfim(12, 12, 256)
    v = VmcSrSymm(w, W.init_symm_params(12, 1, False, 0.01, 3), W.chain_translations(12),
                  prec=prec, graph=True)
    assert kernels(v._eager_step) == v.launches_per_step()


@pytest.mark.parametrize("prec", [FP32, BF16X2])
@pytest.mark.parametrize("ws", [
    [tfim(16, 16, 64), heis(16, 32, 64)], [tfim(100, 100, 64), tfim(70, 70, 64), tfim(20, 20, 64)],
    [heis(64, 64, 64), heis(64, 128, 64), heis(20, 40, 64)], [j1j2(8, 64), heis(64, 64, 64)],
    [tfim(80, 80, 64), heis(64, 64, 64), tfim(16, 64, 64), heis(30, 400, 64), j1j2(8, 64)]],
    ids=["one-tile", "real", "complex", "quads", "mixed"])
def test_batched_iteration(nk, ws, prec):
    from paper_1904_00031_gb300.batch import BatchedVmc
    b = BatchedVmc(ws, prec=prec, graph=True)
    assert kernels(b._eager_step) == b.launches_per_step()
