"""Weight-derivative sums on tensor cores (weight_tc.cu): equal shares of the stages per CTA, against
the FP64 sums, whose values the oracle pins.

Both add the same FP32 tile sums, so a result is as near to FP64 as with whole tasks: the repository's
mixed tolerance for these sums (1e-6 in norm) applies to directions of one sign; a share lost, doubled
or written to another task's rows moves it by 1e-3 or more."""
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


# one piece a task (8,192), a second one of a few stages, more tasks than SMs, a ragged last row
# tile; one group of 32 and of 64 directions, two groups
@pytest.mark.parametrize("n,P", [(8192, 5), (8193, 33), (8300, 5), (9001, 65), (17000, 32), (20001, 70)])
def test_shares(dev, n, P):
    g = synth.random_points(n, seed=n + P, spread=2.0, n_atom=3)
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)
    w = T(np.random.default_rng(P).uniform(0.5, 1.5, size=(P, g.n)) * g.weights)
    eng = vv10.VV10(0)
    eng.prepare(T(g.coords), T(g.weights), T(g.rho), T(g.grad_rho))
    ref = eng.weight_response(w, vv10.VV10_FP64)
    out = eng.weight_response(w, vv10.VV10_MIXED_TF32X3)
    again = eng.weight_response(w, vv10.VV10_MIXED_TF32X3)
    vv10.vv10_sync(eng.h)
    eng.close()
    for name, a, b, c in zip("EUW", ref, out, again):
        assert float((a - b).norm() / a.norm()) <= 1e-6, name
        assert torch.equal(b, c), name
