"""Split-TF32 contraction (hess_tc.cu): equal shares of the stages per CTA, against the FP64 contraction,
whose values the oracle pins.

The same FP32 stage sums are added as with whole tasks, so the repository's mixed tolerance (1e-6 in
norm) applies to trials of one sign; a share lost, doubled or written to another task's rows moves a
result by 1e-3 or more."""
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


# one piece a task (8,192), a second of a few stages, a ragged last row tile, more tasks than SMs; each
# width of a launch, both kinds in one tile (up to 64) and apart, two groups
@pytest.mark.parametrize("n,P", [(8192, 5), (8193, 33), (9001, 5), (20001, 32), (17000, 64), (9001, 70), (17000, 97),
                                 (8400, 150), (8300, 190), (9001, 200)])
def test_shares(dev, n, P):
    g = synth.random_points(n, seed=n + P, spread=2.0, n_atom=3)
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)
    f = np.random.default_rng(P).uniform(0.5, 1.5, size=(P, g.n))
    rt, gt = T(f * g.rho), T(f[:, :, None] * g.grad_rho)
    eng = vv10.VV10(0)
    eng.prepare(T(g.coords), T(g.weights), T(g.rho), T(g.grad_rho))
    eng.energy_potential(vv10.VV10_FP64)
    ref = eng.hessian_contract(rt, gt, vv10.VV10_FP64)
    out = eng.hessian_contract(rt, gt, vv10.VV10_MIXED_TF32X3)
    again = eng.hessian_contract(rt, gt, vv10.VV10_MIXED_TF32X3)
    vv10.vv10_sync(eng.h)
    eng.close()
    for name, a, b, c in zip(("f_rho", "f_gamma"), ref, out, again):
        assert float((a - b).norm() / a.norm()) <= 1e-6, name
        assert torch.equal(b, c), name
