"""The unordered-pair sums (pairsum_sym.cu) and the small FP64 kernel (pairsum.cu) against the
row-by-row kernel (fixed with vv10_set_tiles), whose values the oracle tests pin: every mode, at
the edges of their tiles and of their ranges.

Both form the same FP32 sum over each 256-point tile and add the tiles in FP64 (rows) or
double-FP32 (columns: 2^-47 per tile at most), so the mixed results may differ by a few hundred
tiles x 2^-47 < 4e-12 of the sums; in FP64 a sum of n terms in another order differs by less
than n 2^-53 < 2e-12 for the sizes here.  f^rho, f^gamma and the contraction's diagonal cancel
a digit or two: 1e-9 covers them."""
import numpy as np
import pytest
import torch

from paper_2208_14639_gb300 import synth, vv10

pytestmark = pytest.mark.gpu
FP64, MIXED = vv10.VV10_FP64, vv10.VV10_MIXED_TF32X3
TOL = 1e-9


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    vv10.load(build_if_missing=True)
    return torch.device("cuda", 0)


def results(g, prec, classic, dev):
    T = lambda a, dt=torch.float64: torch.from_numpy(np.ascontiguousarray(a)).to(dev, dt)
    eng = vv10.VV10(0)
    eng.prepare(T(g.coords), T(g.weights), T(g.rho), T(g.grad_rho), T(g.atom_of_point, torch.int32),
                g.molecule.n_atom)
    if classic:
        for mode in range(3):
            vv10.vv10_set_tiles(eng.h, mode + 3 * (prec == FP64), 1, 0)
    rt, gt = T(0.1 * g.rho)[None], T(0.1 * g.grad_rho)[None]
    out = list(eng.energy_potential(prec)) + list(eng.hessian_contract(rt, gt, prec))  # EUW, ABC
    out += list(eng.coord_grad(prec)[:2])                                              # GRAD
    vv10.vv10_set_options(eng.h, vv10.VV10_OPT_FUSE_HESSIAN_SUMS)
    out += list(eng.energy_potential(prec)) + list(eng.hessian_contract(rt, gt, prec))  # EUWABC
    out += [x for x in eng.evaluate(prec, rt, gt)[:7]]                                  # EUWABCG
    again = list(eng.energy_potential(prec))
    assert all(torch.equal(torch.as_tensor(a), torch.as_tensor(b)) for a, b in zip(again, out[7:10]))
    eng.close()
    return [torch.as_tensor(x, dtype=torch.float64).cpu() for x in out]


# FP64: one tile and one point past a tile, both sides of the rule at 4,096, fewer and more rows per
# lane, odd and even tile counts (the half turn); mixed: the smallest size of the rule, and odd and
# even tile counts.
@pytest.mark.parametrize("prec,n", [(FP64, n) for n in (1, 129, 255, 256, 257, 1025, 4096, 4097, 4352, 4353, 4609, 6000)] +
                         [(MIXED, n) for n in (8193, 8448, 8449, 8705, 9900)])
def test_unordered_pairs_match_rows(dev, prec, n):
    g = synth.random_points(n, seed=n, n_atom=3)
    for a, b in zip(results(g, prec, False, dev), results(g, prec, True, dev)):
        scale = torch.maximum(b.abs(), (b.norm() / max(1.0, b.numel()) ** 0.5).expand_as(b))
        assert float(((a - b).abs() / scale.clamp_min(1e-300)).max()) <= TOL


def test_column_sums_in_several_launches(dev):
    """130,000 points: the nine sums' columns do not fit the scratch at once."""
    g = synth.random_points(130_000, seed=5, spread=6.0, n_atom=4)
    for a, b in zip(results(g, MIXED, False, dev), results(g, MIXED, True, dev)):
        assert float((a - b).norm()) <= TOL * float(b.norm())
