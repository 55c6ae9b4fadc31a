"""FP64 tensor-core contraction (hess_o64.cu): the widths of a launch (32, 48 and 64 trials) and the
equal shares of stages per CTA, against the FP64 SIMT contraction, whose values the oracle pins.

Both sum the same products; the tiles of the tensor-core path carry about 46 bits and its results
meet 1e-11 of the SIMT kernel's in norm (test_parity_gpu.py); a misplaced share, trial or factor
moves them by far more."""
import numpy as np
import pytest
import torch

from paper_2208_14639_gb300 import synth, vv10

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    vv10.load(build_if_missing=True)
    return torch.device("cuda", 0)


# points below and above the rule for shares, rows past the last full tile; one launch of each
# width at its edges, and two launches
@pytest.mark.parametrize("n,P", [(1000, 33), (2049, 1), (2049, 32), (3000, 33), (3000, 48), (3000, 49), (3000, 64), (2500, 65)])
def test_launch_widths_and_shares(dev, n, P):
    g = synth.random_points(n, seed=n + P, spread=4.0, n_atom=3)
    T = lambda a, dt=torch.float64: torch.from_numpy(np.ascontiguousarray(a)).to(dev, dt)
    rng = np.random.default_rng(P)
    rt = T(rng.normal(size=(P, g.n)) * g.rho)
    gt = T(rng.normal(size=(P, g.n, 3)) * np.abs(g.grad_rho))
    eng = vv10.VV10(0)
    eng.prepare(T(g.coords), T(g.weights), T(g.rho), T(g.grad_rho))
    eng.energy_potential(vv10.VV10_FP64)
    ref = eng.hessian_contract(rt, gt, vv10.VV10_FP64)
    out = eng.hessian_contract(rt, gt, vv10.VV10_FP64_TC)
    again = eng.hessian_contract(rt, gt, vv10.VV10_FP64_TC)
    vv10.vv10_sync(eng.h)
    eng.close()
    for x, y, z in zip(out, ref, again):
        assert torch.equal(x, z)
        err = (x - y).norm(dim=1) / y.norm(dim=1).clamp_min(1e-300)  # trial by trial
        assert float(err.max()) <= 1e-11
