"""The basis-derivative products of vv10_fock_derivative (K^c of Sec. II.B's F^A) on all-electron
exponents, against sums in wider precision (numpy longdouble).

Every direction array is zero, so that the result is the derivative of the basis functions alone:
X + X^T, X = K^c(A) - [mu on A] K^c(all).  With an s function of an oxygen core the products' factors
span many orders of magnitude over the points, and only one factor of a product carries the
quadrature weight.  Every element is held to 5e-15 of its sum of absolute terms: FP64 FMA chains of
some 500 terms and 64 splits round to sqrt(534) 2^-53 = 2.6e-15 of it, the factors to a few 2^-53
more; factors cut relative to their largest neighbour are off by up to 1e-9 of it."""
import numpy as np
import pytest
import torch

from paper_2208_14639_gb300 import synth, vv10

pytestmark = pytest.mark.gpu


def reference(g, keep, phi, dphi, d2phi, bf_atom, vr, vg):
    """(result, sums of absolute terms), (3 n_atom, nbf, nbf)."""
    L = lambda a: np.asarray(a, dtype=np.longdouble)[keep]
    w, phi, dphi, d2phi = L(g.weights), L(phi), L(dphi), L(d2phi)
    own = g.atom_of_point[keep]
    al, b = (w * L(vr))[:, None], 2 * (w * L(vg))[:, None] * L(g.grad_rho)
    dot = lambda x, y: np.einsum("kd,kmd->km", x, y)

    def build(al, b, phi, dphi, d2phi, sign):
        right = al * phi + dot(b, dphi)
        out = []
        for A in range(g.molecule.n_atom):
            for c in range(3):
                left, second = dphi[:, :, c], dot(b, d2phi[:, :, c, :])
                K = lambda s: left[s].T @ right[s] + second[s].T @ phi[s]
                X = K(own == A) + sign * np.where(bf_atom[:, None] == A, K(own >= 0), 0)
                out.append(X + X.T)
        return np.stack(out)

    return (build(al, b, phi, dphi, d2phi, -1),
            build(abs(al), abs(b), abs(phi), abs(dphi), abs(d2phi), 1))


@pytest.mark.parametrize("order", ["grid", "shuffled"])
@pytest.mark.parametrize("exponent", [9.0, 2266.0, 15330.0, 116506.0])
def test_core_exponents(exponent, order, monkeypatch):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    vv10.load(build_if_missing=True)
    dev = torch.device("cuda", 0)
    T = lambda a, dt=torch.float64: torch.from_numpy(np.ascontiguousarray(a)).to(dev, dt)
    monkeypatch.setitem(synth.AO_SHELLS, "O", list(synth.AO_SHELLS["O"]) + [(0, exponent)])
    mol = synth.water()
    g, phi, dphi, d2phi, basis = synth.ao_moving_system(mol, 30, 110, seed=3, rho_min=-1.0)[:5]
    if order == "shuffled":
        p = np.random.default_rng(1).permutation(g.n)
        g = synth.GridDensity(g.coords[p], g.weights[p], g.rho[p], g.grad_rho[p], g.atom_of_point[p], mol)
        phi, dphi, d2phi = phi[p], dphi[p], d2phi[p]
    vr, vg = -0.1 * np.cbrt(g.rho), 1e-3 / (1.0 + g.rho)
    P = 3 * mol.n_atom
    Z = torch.zeros(P, g.n, dtype=torch.float64, device=dev)
    eng = vv10.VV10(0)
    try:
        eng.prepare(T(g.coords), T(g.weights), T(g.rho), T(g.grad_rho), T(g.atom_of_point, torch.int32), mol.n_atom)
        got = eng.fock_derivative(T(phi), T(dphi), T(d2phi), T(basis.atom, torch.int32), T(vr), T(vg), Z, Z,
                                  torch.zeros(P, g.n, 3, dtype=torch.float64, device=dev), Z, Z, Z, Z,
                                  torch.zeros(3, g.n, mol.n_atom, 3, dtype=torch.float64, device=dev)).cpu().numpy()
    finally:
        eng.close()
    ref, size = reference(g, g.rho >= 1e-10, phi, dphi, d2phi, basis.atom, vr, vg)
    assert (np.abs(got - ref) <= 5e-15 * size).all()
