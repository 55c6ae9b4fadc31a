"""The AO assembly's tensor-core product (gemm_slices.cu) against wider sums (numpy longdouble), held to
what eight slices leave, so that a lost or mis-weighted low slice shows.

In a block of 128 points, with S the power of two of a row's largest element there, the products that
are not formed have an rms of sqrt(7) 74^2 2^-74 < 2^-60 S_a S_b (digits uniform in +-128), the cuts
2^-62 each; the lowest level that is formed is 2^8 larger.  Eight rms of 128 independent terms a block
are allowed, plus rounding: two of the running sums a block, four of every Z, one of the result,
each 2^-53 / sqrt(3) rms, eight rms of these too."""
import numpy as np
import pytest
import torch

from paper_2208_14639_gb300 import synth, vv10

pytestmark = pytest.mark.gpu
U = 2.0**-53 / 3.0**0.5


def bound(phi, z):
    """Allowed error of phi^T z, element by element."""
    cut = run = 0.0
    total = np.zeros((phi.shape[1], z.shape[1]))
    for k in range(0, len(phi), 128):
        a, b = phi[k:k + 128], z[k:k + 128]
        S = lambda x: 2.0 ** np.floor(np.log2(np.maximum(np.abs(x).max(0), 1e-300)))
        cut = cut + 128 * (2.0**-60 * S(a)[:, None] * S(b)[None, :]) ** 2
        part = a.T @ b
        total += part
        run = run + 2 * (U * np.maximum(np.abs(part), np.abs(total))) ** 2
    forming = 4 * U**2 * (phi**2).T @ z**2
    return 8 * np.sqrt(cut + run + forming), total


@pytest.mark.parametrize("n,nbf", [(640, 5), (2000, 40), (5000, 78)])
def test_eight_slices(n, nbf):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    vv10.load(build_if_missing=True)
    dev = torch.device("cuda", 0)
    g = synth.random_points(n, seed=n, n_atom=2)
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev, torch.float64)
    rng = np.random.default_rng(nbf)
    phi, dphi, vr, vg = (rng.normal(size=s) for s in ((n, nbf), (n, nbf, 3), n, n))
    rho = np.maximum(g.rho, 1e-3)
    eng = vv10.VV10(0)
    try:
        assert eng.prepare(T(g.coords), T(g.weights), T(rho), T(g.grad_rho)) == n
        F = eng.fock_matrix(T(phi), T(dphi), T(vr), T(vg)).cpu().numpy()
    finally:
        eng.close()
    L = lambda a: a.astype(np.longdouble)
    z = L(g.weights)[:, None] * (L(vr)[:, None] * L(phi) / 2
                                 + 2 * np.einsum("kc,kmc->km", L(vg)[:, None] * L(g.grad_rho), L(dphi)))
    m = L(phi).T @ z
    tol, _ = bound(phi, z.astype(np.float64))
    ref = m + m.T
    assert (np.abs(F - ref) <= tol + tol.T + 8 * U * np.abs(ref)).all()
