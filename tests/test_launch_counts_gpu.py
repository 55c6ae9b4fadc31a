"""vv10_profile_read's launch counts against the kernel nodes of the captured call: every call whose
kernels were split, joined or replaced, on both sides of the rules that choose between kernels."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2208_14639_gb300 import synth, vv10

pytestmark = pytest.mark.gpu
FP64, TF32, F16, FP64_TC = vv10.VV10_FP64, vv10.VV10_MIXED_TF32X3, vv10.VV10_MIXED_F16X3, vv10.VV10_FP64_TC


def kernel_nodes(graph) -> int:
    cu = ctypes.CDLL("libcuda.so.1")
    g, n = ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t(0)
    assert cu.cuGraphGetNodes(g, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(g, nodes, ctypes.byref(n)) == 0
    kernels = 0
    for node in nodes:
        t = ctypes.c_int(-1)
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(t)) == 0
        kernels += t.value == 0  # CU_GRAPH_NODE_TYPE_KERNEL
    return kernels


CALLS = {}
for _n, _p in ((500, FP64), (5000, FP64), (3000, TF32), (11000, TF32)):
    CALLS[f"energy_{_n}_{_p}"] = (_n, lambda s, p=_p: vv10.vv10_energy_potential(s.h, p, s.a, s.b, None, False))
for _n, _P, _p in ((500, 3, FP64), (3000, 3, FP64_TC), (1000, 3, FP64_TC), (3000, 70, FP64_TC), (9000, 54, TF32),
                   (9000, 100, TF32), (3000, 54, F16), (3000, 200, F16)):
    CALLS[f"contract_{_n}_{_P}_{_p}"] = (_n, lambda s, P=_P, p=_p: vv10.vv10_hessian_contract(
        s.h, p, s.rt[:P], s.gt[:P], s.out[:P], s.out2[:P]))
for _P in (3, 54, 100):
    CALLS[f"weights_9000_{_P}"] = (9000, lambda s, P=_P: vv10.vv10_weight_response(
        s.h, TF32, s.rt[:P], s.out[:P], s.out2[:P], None))
for _n in (400, 3000):
    CALLS[f"fock_{_n}"] = (_n, lambda s: vv10.vv10_fock_matrix(s.h, s.phi, s.dphi, s.a, s.b, s.F[0]))
    CALLS[f"orbital_hessian_{_n}"] = (_n, lambda s: vv10.vv10_orbital_hessian(
        s.h, s.phi, s.dphi, s.rt[:4], s.rt[4:8], s.gt[:4], s.b, s.F))


class State:
    def __init__(self, n, dev):
        g = synth.random_points(n, seed=n, n_atom=2)
        T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev, torch.float64)
        Z = lambda *s: torch.zeros(*s, dtype=torch.float64, device=dev)
        self.eng = vv10.VV10(0)
        self.h = self.eng.h
        self.eng.prepare(T(g.coords), T(g.weights), T(g.rho), T(g.grad_rho))
        self.eng.energy_potential(FP64)
        gen = torch.Generator().manual_seed(1)
        R = lambda *s: torch.randn(*s, dtype=torch.float64, generator=gen).to(dev)
        self.rt, self.gt, self.out, self.out2 = R(200, n), R(200, n, 3), Z(200, n), Z(200, n)
        self.a, self.b, self.phi, self.dphi, self.F = Z(n), Z(n), R(n, 11), R(n, 11, 3), Z(4, 11, 11)


@pytest.mark.parametrize("name", CALLS)
def test_counts(name):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    vv10.load(build_if_missing=True)
    n, call = CALLS[name]
    s = State(n, torch.device("cuda", 0))
    call(s)  # the buffers, and the sums that later calls find
    vv10.vv10_profile_read(s.h)
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call(s)
    counted = {k: v[1] for k, v in vv10.vv10_profile_read(s.h).items() if v[1]}
    nodes = kernel_nodes(graph)
    s.eng.close()
    assert sum(counted.values()) == nodes, counted
