"""NaN, infinities and values whose products leave FP64's range in the AO assembly's tensor-core
product (gemm_slices.cu): they end up in the elements of F and G^t in which a product formed in FP64,
term by term, has them, with zero partners too, and every other element keeps its accuracy (1e-12
of its sum of absolute terms, n 2^-53 for the 1,500 points here, as in test_gemm_slices_gpu.py)."""
import numpy as np
import pytest
import torch

from paper_2208_14639_gb300 import synth, vv10

pytestmark = pytest.mark.gpu
N, NBF, TOL = 1500, 6, 1e-12
NAN, INF = float("nan"), float("inf")


def plant(name, phi, dphi, s):
    if name == "nan_phi":
        phi[700, 2] = NAN
    elif name == "nan_phi_zero_partners":
        phi[700, :] = 0.0
        dphi[700] = 0.0
        phi[700, 2] = NAN
    elif name == "inf_phi":
        phi[701, 1] = INF
    elif name == "inf_phi_small_partners":
        phi[701, :] *= 1e-30
        dphi[701] *= 1e-30
        phi[701, 1] = -INF
    elif name == "nan_gradient":
        dphi[3, 4, 1] = NAN
    elif name == "nan_scalar":
        s[0, 1499] = NAN
    elif name == "inf_scalar_zero_partner":
        phi[130, 3] = 0.0
        dphi[130, 3] = 0.0
        s[-1, 130] = INF
    elif name == "both_infinities":
        phi[10, 0], phi[900, 0] = INF, -INF
    elif name == "beyond_the_range":
        f = torch.logspace(-90, 250, NBF, dtype=torch.float64, device=phi.device)
        phi *= f
        dphi *= f[:, None]
    return phi, dphi, s


@pytest.mark.parametrize("trials", [0, 3], ids=["fock", "orbital_hessian"])
@pytest.mark.parametrize("name", ["nan_phi", "nan_phi_zero_partners", "inf_phi", "inf_phi_small_partners", "nan_gradient",
                                  "nan_scalar", "inf_scalar_zero_partner", "both_infinities", "beyond_the_range"])
def test_as_an_fp64_product(name, trials):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    vv10.load(build_if_missing=True)
    dev = torch.device("cuda", 0)
    g = synth.random_points(N, seed=5, n_atom=2)
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev, torch.float64)
    gen = torch.Generator().manual_seed(1)
    R = lambda *s: torch.randn(*s, dtype=torch.float64, generator=gen).to(dev)
    P = max(trials, 1)
    w, rho, grad = T(g.weights), torch.clamp(T(g.rho), min=1e-3), T(g.grad_rho)  # every point is kept
    phi, dphi, s = plant(name, R(N, NBF), R(N, NBF, 3), R(P, N))
    fg, vg, gt = R(P, N), R(N), R(P, N, 3)
    eng = vv10.VV10(0)
    try:
        assert eng.prepare(T(g.coords), w, rho, grad) == N
        if trials:
            got = eng.orbital_hessian(phi, dphi, s, fg, gt, vg)
            v = fg[:, :, None] * grad + vg[:, None] * gt
        else:
            got = eng.fock_matrix(phi, dphi, s[0], fg[0])[None]
            v = fg[:, :, None] * grad
        torch.cuda.synchronize()
    finally:
        eng.close()
    planted = 0
    for t in range(P):
        # the coefficients times phi and grad phi, so that a NaN or an infinity meets every zero
        z = w[:, None] * (0.5 * s[t][:, None] * phi + (2.0 * v[t][:, None, :] * dphi).sum(-1))
        m = (phi[:, :, None] * z[:, None, :]).sum(0)
        ref = m + m.T
        fin = torch.isfinite(ref)
        planted += int((~fin).sum())
        size = (phi.abs()[:, :, None] * z.abs()[:, None, :]).sum(0)
        size = size + size.T
        # an overflowing sum is an infinity or NaN by the order of its terms
        sure = torch.isfinite(size) if name == "beyond_the_range" else torch.ones_like(fin)
        assert torch.equal(torch.isnan(got[t])[sure], torch.isnan(ref)[sure])
        inf = torch.isinf(ref) & sure
        assert torch.equal(got[t][inf], ref[inf]) and torch.isfinite(got[t][fin & sure]).all()
        ok = fin & torch.isfinite(size)
        assert ((got[t] - ref).abs()[ok] <= TOL * size[ok]).all()
    assert planted > 0
