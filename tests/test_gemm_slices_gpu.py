"""The AO assembly's tensor-core product (gemm_slices.cu) through vv10_fock_matrix, against FP64
torch on the same arrays: edges of the 128 x 64 tile and of the 128-point block, short products on
either side of the rule, and columns of very different magnitude.

The product is exact to 2^-60 of each block's largest terms and rounded twice per block; the FP64
matmul it is compared with rounds at every point: n 2^-53 of sum |a b| at most, 1e-12 for the
sizes here, and every entry is held to that of its row's and column's magnitude."""
import numpy as np
import pytest
import torch

from paper_2208_14639_gb300 import synth, vv10

pytestmark = pytest.mark.gpu
TOL = 1e-12


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    vv10.load(build_if_missing=True)
    return torch.device("cuda", 0)


def fock_and_reference(dev, n, nbf, spread):
    g = synth.random_points(n, seed=n, n_atom=2)
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev, torch.float64)
    eng = vv10.VV10(0)
    w, rho, grad = T(g.weights), T(g.rho), T(g.grad_rho)
    eng.prepare(T(g.coords), w, rho, grad)
    gen = torch.Generator(device="cpu").manual_seed(nbf)
    R = lambda *s: torch.randn(*s, dtype=torch.float64, generator=gen).to(dev)
    scale = 10.0 ** (spread * (2.0 * torch.rand(nbf, dtype=torch.float64, generator=gen) - 1.0)).to(dev)
    # magnitudes that vary over the points too, as basis functions on a grid do
    phi = R(n, nbf) * torch.exp(-4.0 * R(n, nbf).abs()) * scale
    dphi = R(n, nbf, 3) * torch.exp(-4.0 * R(n, nbf, 1).abs()) * scale[:, None]
    vr, vg = R(n), R(n)
    F = eng.fock_matrix(phi, dphi, vr, vg)
    vv10.vv10_sync(eng.h)
    eng.close()
    keep = rho >= 1e-10
    phi, dphi = phi[keep], dphi[keep]
    z = w[keep][:, None] * (0.5 * vr[keep][:, None] * phi
                            + 2.0 * torch.einsum("kc,kmc->km", (vg[:, None] * grad)[keep], dphi))
    m, size = phi.T @ z, phi.abs().T @ z.abs()
    return F, m + m.T, size + size.T


@pytest.mark.parametrize("n,nbf", [(300, 5), (511, 64), (512, 1), (513, 63), (640, 65), (641, 128), (1000, 130), (5000, 78)])
def test_product_matches_fp64(dev, n, nbf):
    F, ref, size = fock_and_reference(dev, n, nbf, 0.0)
    assert float(((F - ref).abs() / size).max()) <= TOL


def test_columns_of_any_magnitude(dev):
    F, ref, size = fock_and_reference(dev, 2000, 40, 100.0)
    assert torch.isfinite(F).all()
    assert float(((F - ref).abs() / size).max()) <= TOL
    assert torch.equal(F, F.T)
