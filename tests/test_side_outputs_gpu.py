"""The side outputs of the equal shares (split-TF32 and FP64 tensor-core contractions, weight-derivative
sums): a later call with less work, or in another precision, leaves the buffers in place that a
captured graph uses, and a call that finds no room for them deals whole tasks.

9,000 points: 54 directions are dealt in equal shares, 100 in whole tasks.  Replays run the captured
kernels on unchanged inputs: the same bits.  Shares and whole tasks end the FP32 sums at the same
stages and add them in FP64 in another order (1e-12); the FP64 tensor-core contraction's
double-FP32 sums end elsewhere (2^-46 each, 1e-11 in norm, as the header states)."""
import numpy as np
import pytest
import torch

from paper_2208_14639_gb300 import synth, vv10

pytestmark = pytest.mark.gpu
FP64, TF32, F16, FP64_TC = vv10.VV10_FP64, vv10.VV10_MIXED_TF32X3, vv10.VV10_MIXED_F16X3, vv10.VV10_FP64_TC
N = 9000
SIDE = 152 * 192 * 128 * 8


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    vv10.load(build_if_missing=True)
    return torch.device("cuda", 0)


class Setup:
    def __init__(self, dev, prec):
        self.dev, self.prec = dev, prec
        self.g = synth.random_points(N, seed=9, n_atom=3)
        T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev, torch.float64)
        self.eng = vv10.VV10(0)
        assert self.eng.prepare(T(self.g.coords), T(self.g.weights), T(self.g.rho), T(self.g.grad_rho)) == N
        self.eng.energy_potential(prec)
        gen = torch.Generator().manual_seed(3)
        R = lambda *s: torch.randn(*s, dtype=torch.float64, generator=gen).to(dev)
        self.rt, self.gt, self.w = R(100, N) * T(self.g.rho), R(100, N, 3) * T(self.g.grad_rho).abs(), R(100, N)

    def contract(self, P, prec=None, out=None):
        out = out or [torch.empty(P, N, dtype=torch.float64, device=self.dev) for _ in range(2)]
        vv10.vv10_hessian_contract(self.eng.h, self.prec if prec is None else prec, self.rt[:P], self.gt[:P], *out)
        return out

    def weights(self, P, out=None):
        out = out or [torch.empty(P, N, dtype=torch.float64, device=self.dev) for _ in range(3)]
        vv10.vv10_weight_response(self.eng.h, self.prec, self.w[:P], *out)
        return out


def replays(setup, call, later):
    """The outputs of `call` outside a capture and replayed after `later`."""
    ref = [x.clone() for x in call(None)]
    out = [torch.empty_like(x) for x in ref]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call(out)
    later()
    for x in out:
        x.fill_(float("nan"))
    graph.replay()
    torch.cuda.synchronize()
    return all(torch.equal(a, b) for a, b in zip(ref, out))


def test_graph_of_more_trials(dev):
    s = Setup(dev, TF32)
    assert replays(s, lambda o: s.contract(100, out=o), lambda: s.contract(54))
    s.eng.close()


def test_graph_of_more_weight_directions(dev):
    s = Setup(dev, TF32)
    assert replays(s, lambda o: s.weights(100, out=o), lambda: s.weights(54))
    s.eng.close()


def test_graph_of_another_precision(dev):
    s = Setup(dev, F16)
    s.contract(54)
    assert replays(s, lambda o: s.contract(54, out=o), lambda: s.contract(54, TF32))
    s.eng.energy_potential(FP64)
    s.contract(1, FP64)  # the diagonal's sums in FP64 for every later call
    assert replays(s, lambda o: s.contract(54, out=o), lambda: s.contract(54, FP64_TC))
    s.eng.close()


def refused(call, k):
    """`call` with its k-th device allocation refused, and again."""
    a = [x.clone() for x in call(k)]
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    b = call(0)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] >= 0.9 * SIDE  # it was the side outputs' allocation
    return a, b


@pytest.mark.parametrize("what,tol", [("contract", 1e-12), ("weights", 1e-12), ("fp64_tc", 1e-11)])
def test_no_room(dev, what, tol):
    s = Setup(dev, FP64 if what == "fp64_tc" else TF32)
    out = [torch.empty(54, N, dtype=torch.float64, device=dev) for _ in range(3)]

    def call(k):
        vv10.vv10_debug_inject(s.eng.h, vv10.VV10_DEBUG_FAIL_ALLOC, k)
        if what == "weights":
            return s.weights(54, out)
        return s.contract(54, FP64_TC if what == "fp64_tc" else TF32, out[:2])

    # larger buffers than the call needs are in place, but for the FP64 slices' three
    s.weights(100) if what == "weights" else s.contract(100)
    a, b = refused(call, 4 if what == "fp64_tc" else 1)
    for x, y in zip(a, b):
        assert float((x - y).norm()) <= tol * float(y.norm())
    s.eng.close()
