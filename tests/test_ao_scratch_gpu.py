"""vv10_orbital_hessian's scratch with few basis functions: about 1 GB for the per-trial operands, as the
header states, also where a trial's coefficients are larger than its operand (one function: 4 : 1).

Channels on both sides of the chunks' edges against FP64 torch: n 2^-53 of the sum of absolute terms."""
import numpy as np
import pytest
import torch

from paper_2208_14639_gb300 import synth, vv10

pytestmark = pytest.mark.gpu


def test_one_function_many_trials():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    vv10.load(build_if_missing=True)
    dev = torch.device("cuda", 0)
    n, P = 200_000, 1000
    g = synth.random_points(n, seed=4, spread=6.0)
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev, torch.float64)
    w, rho, grad = T(g.weights), torch.clamp(T(g.rho), min=1e-3), T(g.grad_rho)
    gen = torch.Generator(device=dev).manual_seed(2)
    R = lambda *s: torch.randn(*s, dtype=torch.float64, device=dev, generator=gen)
    phi, dphi, f_rho, f_gamma, grad_t, vg = R(n, 1), R(n, 1, 3), R(P, n), R(P, n), R(P, n, 3), R(n)
    G = torch.empty(P, 1, 1, dtype=torch.float64, device=dev)
    eng = vv10.VV10(0)
    try:
        assert eng.prepare(T(g.coords), w, rho, grad) == n
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        vv10.vv10_orbital_hessian(eng.h, phi, dphi, f_rho, f_gamma, grad_t, vg, G)
        torch.cuda.synchronize()
        assert free - torch.cuda.mem_get_info()[0] <= 1.5 * 2**30
    finally:
        eng.close()
    for t in (0, 40, 41, 42, 670, 671, P - 1):
        v = f_gamma[t][:, None] * grad + vg[:, None] * grad_t[t]
        terms = 2.0 * phi[:, 0] * w * (0.5 * f_rho[t] * phi[:, 0] + 2.0 * (v * dphi[:, 0]).sum(-1))
        size = 2.0 * phi[:, 0].abs() * w * (0.5 * (f_rho[t] * phi[:, 0]).abs() + 2.0 * (v * dphi[:, 0]).abs().sum(-1))
        assert abs(float(G[t, 0, 0] - terms.sum())) <= n * 2.0**-53 * float(size.sum())
