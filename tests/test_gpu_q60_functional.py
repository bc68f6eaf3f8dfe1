"""The fixed-point and series forms of the plaquette, the functional and its gradient against FP64 torch and
the oracle, on both sides of each of their rules: norms of omega where the series are doubled or left for the
eigenvectors, links that are not near SU(3), and values that are not finite."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

DIMS = (6, 4, 5, 3)


def lambdas():
    g = np.zeros((8, 3, 3), np.complex128)
    for k, (i, j) in ((0, (0, 1)), (3, (0, 2)), (5, (1, 2))):
        g[k][i, j] = g[k][j, i] = 1
        g[k + 1][i, j], g[k + 1][j, i] = -1j, 1j
    g[2] = np.diag([1, -1, 0])
    g[7] = np.diag([1, 1, -2]) / np.sqrt(3)
    return g


def reference(U, w):
    """F and dF/domega in torch float64 (eigenvectors of omega by torch.linalg.eigh)."""
    import torch
    om = torch.tensor(w.reshape(U.shape[1:5] + (8,)), requires_grad=True)
    H = torch.einsum("...a,aij->...ij", om.to(torch.complex128), torch.tensor(lambdas() / 2))
    g = torch.linalg.matrix_exp(1j * H)
    F = 0
    for mu in range(4):
        F = F + torch.einsum("...ij,...jk,...ik->", g, torch.tensor(U[mu]), torch.roll(g, -1, 3 - mu).conj()).real
    F = F / (12.0 * U[0, ..., 0, 0].size)
    grad, = torch.autograd.grad(F, om)
    return float(F), grad.numpy().reshape(-1, 8)


# norms of omega are 2 * size: no doubling, doublings, eigenvectors
@pytest.mark.parametrize("size", [0.0, 1e-9, 0.02, 0.2, 0.26, 1.0, 7.0, 31.0, 33.0, 60.0])
@pytest.mark.parametrize("links", ["su3", "scaled"])
def test_functional_and_gradient(size, links):
    import paper_1210_8018_gb300 as lgf
    U = synth.config(DIMS, 71, 0.6)
    if links == "scaled":  # out of the fixed-point range for the links of one time slice
        U[:, 1] *= 1.7
    rng = np.random.default_rng(72)
    V = U[0, ..., 0, 0].size
    w = rng.standard_normal((V, 8))
    w *= 2 ** 0.5 * 2 * size / np.linalg.norm(w, axis=1, keepdims=True)
    if size:
        w[5] = 0
        w[6, :7] = 0  # two equal eigenvalues
    F0, g0 = reference(U, w)
    with lgf.Lattice(DIMS) as lat:
        gm = np.empty(U.shape[1:], np.complex128)
        F = lat.functional(U, w, gm)
        grad = np.empty((V, 8))
        lat.functional_grad(U, w, grad)
    # both sides lose about eps |omega| in the phases of exp(i omega); the reference's own Pade squaring too
    tol = 1e-14 * (1 + 4 * size)
    assert abs(F - F0) < tol
    assert np.abs(gm @ gm.conj().swapaxes(-1, -2) - np.eye(3)).max() < 10 * tol
    assert np.abs(grad - g0).max() * V < 10 * tol


def test_functional_not_finite():
    import paper_1210_8018_gb300 as lgf
    U = synth.config(DIMS, 73, 0.6)
    V = U[0, ..., 0, 0].size
    w = np.full((V, 8), 0.01)
    w[7, 3] = np.nan
    grad = np.empty((V, 8))
    with lgf.Lattice(DIMS) as lat:
        assert not np.isfinite(lat.functional(U, w))
        lat.functional_grad(U, w, grad)
    assert np.isnan(grad[7]).all() and np.isnan(grad[8]).all() and np.isfinite(grad[40]).all()


def exact_measures(U):
    """theta, F and the plaquette, summed in extended precision (a serial sum in double is too coarse)."""
    n = 3 * U[0, ..., 0, 0].size
    D = oracle.delta(U)
    theta = (np.abs(D) ** 2).astype(np.longdouble).sum() / n
    F = np.trace(U, axis1=-2, axis2=-1).real.astype(np.longdouble).sum() / (4 * n)
    p = np.longdouble(0)
    for mu in range(4):
        for nu in range(mu + 1, 4):
            a = U[mu] @ np.roll(U[nu], -1, 3 - mu)
            b = U[nu] @ np.roll(U[mu], -1, 3 - nu)
            p += (a * b.conj()).real.astype(np.longdouble).sum()
    return theta, F, p / (6 * n)


@pytest.mark.parametrize("dims", [DIMS, (16, 8, 8, 8), (9, 5, 4, 10)])
@pytest.mark.parametrize("factor", [1.0, 0.3, 1.7, 70.0])
def test_measure(dims, factor):
    """SU(3) links and links small enough take the fixed-point pass, larger ones the FP64 kernels."""
    import paper_1210_8018_gb300 as lgf
    U = synth.config(dims, 74, 0.5)
    U[2, 1] *= factor if factor < 64 else 1.0
    with lgf.Lattice(dims) as lat:
        if factor > 64:
            U[1, 0, 0, 0, 0, 1, 1] = np.nan
            r = lat.measure(U)
            assert not np.isfinite(r["F"]) and not np.isfinite(r["plaquette"])
            return
        r = lat.measure(U)
    theta, F, plaq = exact_measures(U)
    assert abs(r["theta"] - theta) < 2e-15 * max(1.0, r["theta"])
    assert abs(r["F"] - F) < 1e-15
    assert abs(r["plaquette"] - plaq) < 1e-15 * max(1.0, factor ** 2)
