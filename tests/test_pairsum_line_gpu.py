"""The mixed pair sums on both sides of the line between the row-by-row and the unordered-pair kernel
(10,752 points): which one runs, by the reduction that the latter adds, and beyond the line the row
kernel's values in every mode, at the smallest sizes and odd and even tile counts, with
test_pairsum_sym_gpu.py's bound."""
import numpy as np
import pytest
import torch

from paper_2208_14639_gb300 import synth, vv10
from test_pairsum_sym_gpu import MIXED, TOL, results

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    vv10.load(build_if_missing=True)
    return torch.device("cuda", 0)


@pytest.mark.parametrize("n,reductions", [(9000, 0), (10752, 0), (10753, 1), (12000, 1)])
def test_kernel_of_a_size(dev, n, reductions):
    g = synth.random_points(n, seed=n)
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev, torch.float64)
    eng = vv10.VV10(0)
    try:
        assert eng.prepare(T(g.coords), T(g.weights), torch.clamp(T(g.rho), min=1e-6), T(g.grad_rho)) == n
        for flags in (0, vv10.VV10_OPT_FUSE_HESSIAN_SUMS):
            vv10.vv10_set_options(eng.h, flags)
            vv10.vv10_profile_read(eng.h)
            eng.energy_potential(MIXED)
            assert vv10.vv10_profile_read(eng.h)["energy_epilogue"][1] == 2 + reductions
    finally:
        eng.close()


@pytest.mark.parametrize("n", [10753, 11008, 11009, 11265])
def test_unordered_pairs_beyond_it(dev, n):
    g = synth.random_points(n, seed=n, n_atom=3)
    for a, b in zip(results(g, MIXED, False, dev), results(g, MIXED, True, dev)):
        scale = torch.maximum(b.abs(), (b.norm() / max(1.0, b.numel()) ** 0.5).expand_as(b))
        assert float(((a - b).abs() / scale.clamp_min(1e-300)).max()) <= TOL
