"""The gradient of the functional and the measurements against extended precision where the 60-bit fixed point and
the series could hold less than FP64: fields close to unity, links far from unit length or between the steps of the
fixed point, and the norms of omega at which the series are doubled or left for the eigenvectors."""
import numpy as np
import pytest

import synth
from helpers import gell_mann, identity_links

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


def near_unity(d, seed):
    rng = np.random.default_rng(seed)
    x = d * (rng.normal(size=(4, SITES, 3, 3)) + 1j * rng.normal(size=(4, SITES, 3, 3)))
    return np.ascontiguousarray((np.eye(3) + x - dag(x)).reshape((4,) + DIMS[::-1] + (3, 3))), rng


# eight terms of size d to an element of the staple and three to one of M, whose rounding is that of their size:
# fewer than 64 roundings of 16 d, over 12 V
@pytest.mark.parametrize("omega", [0.0, 1.0])
@pytest.mark.parametrize("d", [1e-12, 1e-9, 1e-6, 1e-3])
def test_near_unity(d, omega):
    U, rng = near_unity(d, 61)
    w = omega * d * rng.normal(size=(SITES, 8))
    err = np.abs(device_gradient(U, w) - gradient(U, w)).max()
    assert err < 64 * 2.0 ** -53 * 16 * d / (12 * SITES), err


def test_one_pair_of_elements_small():
    """Links of an SU(2) subgroup, and the elements that leave it of size 1e-9."""
    U, rng = near_unity(1e-9, 63)
    a = rng.uniform(-3, 3, size=U.shape[:5])
    c, s = np.cos(a), np.sin(a)
    R = np.broadcast_to(np.eye(3, dtype=complex), U.shape).copy()
    R[..., 0, 0], R[..., 0, 1], R[..., 1, 0], R[..., 1, 1] = c, s, -s, c
    U = R @ U
    U[..., 0, 0] *= np.exp(0.3j)
    w = np.zeros((SITES, 8))
    got, ref = device_gradient(U, w), gradient(U, w)
    assert np.abs(got - ref)[:, 3:7].max() < 64 * 2.0 ** -53 * 16e-9 / (12 * SITES)
    assert np.abs(got - ref).max() < 64 * 2.0 ** -53 * 16 / (12 * SITES)


@pytest.mark.parametrize("factor", [2.0 ** -100, 2.0 ** 135, 2.0 ** 500])
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


def test_measure_between_the_steps():
    """Elements below the last step of Delta's fixed point are dropped whatever their sign, as lgf_delta drops them."""
    import paper_1210_8018_gb300 as lgf
    U = identity_links(DIMS)
    U[1, 0, 1, 2, 3, 0, 1] = -2.0 ** -58
    U[2, 1, 0, 1, 2, 1, 1] += -1j * 2.0 ** -58
    with lgf.Lattice(DIMS) as lat:
        theta, _ = lat.delta(U, np.empty(U.shape[1:], complex))
        r = lat.measure(U)
    assert r["theta"] == theta == 0.0
    U = synth.config(DIMS, 69, 0.6)
    with lgf.Lattice(DIMS) as lat:
        theta, _ = lat.delta(U, np.empty(U.shape[1:], complex))
        r = lat.measure(U)
    assert abs(r["theta"] - theta) < 16 * 2.0 ** -53 * theta


def test_measure_of_short_links():
    import paper_1210_8018_gb300 as lgf
    U = synth.config(DIMS, 70, 0.6)
    with lgf.Lattice(DIMS) as lat:
        r, q = lat.measure(U), lat.measure(U * 2.0 ** -100)
    # nine terms to a product, four products, and their sum over the lattice
    assert abs(q["plaquette"] * 2.0 ** 400 - r["plaquette"]) < 64 * 2.0 ** -53
    assert abs(q["F"] * 2.0 ** 100 - r["F"]) < 64 * 2.0 ** -53
