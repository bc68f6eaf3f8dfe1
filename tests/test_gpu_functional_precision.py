"""The gradient of the functional against extended precision: links far beyond the range of a float, and the norms
of omega at which its series are doubled or left for the eigenvectors."""
import numpy as np
import pytest

import synth
from helpers import gell_mann

pytestmark = pytest.mark.gpu

DIMS = (6, 4, 5, 3)
SITES = int(np.prod(DIMS))
LD = np.clongdouble


def mul(a, b):
    return (a[..., :, :, None] * b[..., None, :, :]).sum(-2)


def dag(a):
    return np.swapaxes(a, -1, -2).conj()


def gradient(U, w):
    """-(1/12V) Tr[T^a Y], Y = sum_n (-i ad_omega)^n A / (n+1)!, A = (M - M^+)/(2i), M = g K."""
    T = gell_mann().astype(LD) / 2
    H = (w.astype(LD).reshape(U.shape[1:5] + (8, 1, 1)) * T).sum(-3)
    g = term = np.broadcast_to(np.eye(3, dtype=LD), H.shape)
    for n in range(1, 60):
        term = mul(term, 1j * H) / n
        g = g + term
    K = np.zeros_like(H)
    for mu in range(4):
        u = U[mu].astype(LD)
        K = K + mul(u, dag(np.roll(g, -1, 3 - mu))) + np.roll(dag(mul(g, u)), 1, 3 - mu)
    M = mul(g, K)
    X = (M - dag(M)) / 2j
    Y = np.zeros_like(X)
    f = np.longdouble(1)
    for n in range(60):
        f = f / (n + 1)
        Y = Y + f * X
        X = -1j * (mul(H, X) - mul(X, H))
    return -(T * np.swapaxes(Y[..., None, :, :], -1, -2)).sum((-1, -2)).real.reshape(-1, 8) / (12 * SITES)


def device_gradient(U, w):
    import paper_1210_8018_gb300 as lgf
    out = np.empty((SITES, 8))
    with lgf.Lattice(DIMS) as lat:
        lat.functional_grad(U, w, out)
    return out


@pytest.mark.parametrize("factor", [2.0 ** 135, 2.0 ** 500])
def test_scaled_links(factor):
    U = synth.config(DIMS, 65, 0.6)
    w = 0.1 * np.random.default_rng(66).normal(size=(SITES, 8))
    ref = gradient(U, w)
    err = np.abs(device_gradient(U * factor, w) / factor - ref).max()
    assert err < 64 * 2.0 ** -53 * 16 / (12 * SITES), err


# the error of eigenvectors and of two doublings: a few roundings of 16 (1 + norm)
@pytest.mark.parametrize("norm", [0.5 - 1e-9, 0.5 + 1e-9, 1.0, 2.0 - 1e-9, 2.0 + 1e-9, 3.0 - 1e-9, 3.0 + 1e-9])
def test_norms_beside_the_rules(norm):
    U = synth.config(DIMS, 67, 0.6)
    w = np.random.default_rng(68).normal(size=(SITES, 8))
    w *= 2 ** 0.5 * norm / np.linalg.norm(w, axis=1, keepdims=True)
    err = np.abs(device_gradient(U, w) - gradient(U, w)).max()
    assert err < 64 * 2.0 ** -53 * 16 * (1 + norm) / (12 * SITES), err
