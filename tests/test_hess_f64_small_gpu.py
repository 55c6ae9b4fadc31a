"""FP64 contraction of systems with fewer CTAs than SMs: chunks of trials by the SMs that are free, at the
chunk widths' edges, against the oracle (1e-10 in norm and per element of |ref_i| + rms, as in
test_hess_f64_chunks_gpu.py), and at a size where a wide chunk on few SMs would show."""
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


def system(dev, n, P):
    g = synth.random_points(n, seed=n + P, spread=3.0, n_atom=3)
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)
    rng = np.random.default_rng(P)
    rt = rng.normal(size=(P, g.n)) * g.rho
    gt = rng.normal(size=(P, g.n, 3)) * np.abs(g.grad_rho)
    eng = vv10.VV10(0)
    eng.prepare(T(g.coords), T(g.weights), T(g.rho), T(g.grad_rho))
    eng.energy_potential(vv10.VV10_FP64)
    return g, rt, gt, eng, T(rt), T(gt)


@pytest.mark.parametrize("n,P", [(100, 152), (100, 153), (100, 310), (300, 33), (300, 51), (257, 70), (700, 12), (1000, 33),
                                 (1000, 9), (1500, 54), (2100, 33)])
def test_chunks_by_free_sms(dev, oracle_mod, n, P):
    g, rt, gt, eng, drt, dgt = system(dev, n, P)
    out = eng.hessian_contract(drt, dgt, vv10.VV10_FP64)
    vv10.vv10_sync(eng.h)
    eng.close()
    ref = oracle_mod.hessian_contract(g.coords, g.weights, g.rho, g.grad_rho, rt, gt)
    for a, r, what in zip(out, ref, ("f_rho", "f_gamma")):
        check(a.cpu().numpy(), r, 1e-10, what=what)


def test_a_few_trials_more_are_not_a_wider_cta(dev):
    """1,000 points: 33 trials in CTAs of 36 took over four times a single trial's time."""
    def ms(P):
        _, _, _, eng, rt, gt = system(dev, 1000, P)
        eng.hessian_contract(rt, gt, vv10.VV10_FP64)
        vv10.vv10_profile_enable(eng.h, True)
        vv10.vv10_profile_read(eng.h)
        for _ in range(20):
            eng.hessian_contract(rt, gt, vv10.VV10_FP64)
        t = vv10.vv10_profile_read(eng.h)["contraction_fp64"][0]
        eng.close()
        return t
    assert ms(33) <= 3.2 * ms(1)
