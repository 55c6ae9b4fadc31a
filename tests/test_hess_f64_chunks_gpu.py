"""FP64 contraction (k_hess_f64): trials per CTA from 1 to 40 at their edges, one and two chunks, j splits
of small and larger systems, against the oracle, at the FP64 tolerance of the parity tests (1e-10 in norm
and per element of |ref_i| + rms)."""
import numpy as np
import pytest
import torch

from paper_2208_14639_gb300 import synth, vv10
from parity_util import check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    vv10.load(build_if_missing=True)
    return torch.device("cuda", 0)


@pytest.mark.parametrize("n,P", [(65, 1), (1500, 1), (300, 2), (129, 3), (300, 4), (300, 5), (127, 12), (1500, 13),
                                 (128, 17), (300, 21), (300, 28), (300, 33), (1100, 36), (129, 40), (300, 41),
                                 (64, 80), (200, 81)])
def test_trials_per_cta(dev, oracle_mod, n, P):
    g = synth.random_points(n, seed=n + P, spread=3.0, n_atom=3)
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)
    rng = np.random.default_rng(P)
    rt = rng.normal(size=(P, g.n)) * g.rho
    gt = rng.normal(size=(P, g.n, 3)) * np.abs(g.grad_rho)
    ref = oracle_mod.hessian_contract(g.coords, g.weights, g.rho, g.grad_rho, rt, gt)
    eng = vv10.VV10(0)
    eng.prepare(T(g.coords), T(g.weights), T(g.rho), T(g.grad_rho))
    eng.energy_potential(vv10.VV10_FP64)
    out = eng.hessian_contract(T(rt), T(gt), vv10.VV10_FP64)
    vv10.vv10_sync(eng.h)
    eng.close()
    for a, r, what in zip(out, ref, ("f_rho", "f_gamma")):
        check(a.cpu().numpy(), r, 1e-10, what=what)
