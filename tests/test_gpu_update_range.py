"""The general double update, U' = g(x) U g^+(x+mu) in 60-bit fixed point, beside its rules: links and gauge
matrices whose entries are below 2 but whose rows are not of unit length, whose rows are not orthogonal, that are
short, nearly diagonal, 2 and above or not finite. Every such site lies in a warp of ordinary ones, and every
direction is compared with rows 0-1 by products and row 2 = conj(row0 x row1), both in extended precision."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

DIMS = (8, 4, 4, 4)


def expected(U, g):
    U, g = U.astype(np.clongdouble), g.astype(np.clongdouble)
    out = np.empty_like(U)
    for mu in range(4):
        gf = np.roll(g, -1, 3 - mu)
        t = (g[..., :, :, None] * U[mu][..., None, :, :]).sum(-2)
        out[mu] = (t[..., :, None, :] * gf.conj()[..., None, :, :]).sum(-1)
        r0, r1 = out[mu][..., 0, :], out[mu][..., 1, :]
        for j in range(3):
            a, b = (j + 1) % 3, (j + 2) % 3
            out[mu][..., 2, j] = (r0[..., a] * r1[..., b] - r0[..., b] * r1[..., a]).conj()
    return out


def update(U, g):
    import paper_1210_8018_gb300 as lgf
    U = U.copy()
    with lgf.Lattice(DIMS) as lat:
        lat.update(U, g)
    return U


def check(U, g):
    out, ref = update(U, g), expected(U, g)
    # three-term products twice, then a difference of two: fewer than 32 roundings of numbers of these sizes
    size = np.sqrt((np.abs(ref) ** 2).sum(-1, keepdims=True).astype(float))  # of each row
    bound = np.concatenate([size[..., :2, :], size[..., :1, :] * size[..., 1:2, :] + size[..., 2:, :]], -2)
    big = np.abs(g).max((-1, -2))
    scale = np.stack([big * np.roll(big, -1, 3 - mu) for mu in range(4)]) * np.abs(U).max((-1, -2))
    bound = np.maximum(bound, scale[..., None, None] * np.maximum(1, np.stack([scale] * 3, -1)[..., None] * [[0], [0], [1]]))
    err = np.abs(out - ref).astype(float)
    assert (err <= 32 * 2.0 ** -53 * bound).all(), (err / bound).max()


def fields(seed):
    U = synth.config(DIMS, seed, 0.6)
    g = np.ascontiguousarray(synth.config(DIMS, seed + 1, 0.0)[0])  # random SU(3)
    return U, g


def pick(m, below):
    """Sites whose matrix has every entry's parts below a limit."""
    top = np.maximum(np.abs(m.real), np.abs(m.imag)).max((-1, -2))
    return np.argwhere(top < below)


FLAT = np.full((3, 3), np.exp(0.25j * np.pi) / np.sqrt(3))  # rows and columns of unit length, norm 3^(1/2)


@pytest.mark.parametrize("kind", ["long", "flat", "short", "shorter", "large", "huge"])
@pytest.mark.parametrize("what", ["link", "gauge", "both"])
def test_not_special_unitary(kind, what):
    U, g = fields(51)
    factor = {"long": 2.5, "short": 0.2, "shorter": 1e-9, "large": 7.0, "huge": 1e30}.get(kind)
    for m in ([U[mu] for mu in range(4)] if what != "gauge" else []) + ([g] if what != "link" else []):
        if kind == "flat":
            m[1, 2, 3, 5] = FLAT
            m[2, 0, 1] = FLAT * np.exp(0.5j * np.arange(8))[:, None, None]
        else:
            at = pick(m, 0.79)
            assert len(at) > 3
            for a in at[:3]:
                m[tuple(a)] *= factor
    check(U, g)


def test_not_finite_stays_where_it_is():
    U, g = fields(53)
    ref = update(U, g)
    V = U.copy()
    V[1, 2, 1, 3, 6, 0, 1] = np.nan
    V[3, 0, 1, 3, 6, 2, 2] = np.inf
    out = update(V, g)
    for at in ((1, 2, 1, 3, 6), (3, 0, 1, 3, 6)):
        assert not np.isfinite(out[at]).all()
        out[at] = ref[at]
    assert np.abs(out - ref).max() < 32 * 2.0 ** -53


def test_nearly_diagonal():
    """Elements beside the diagonal of size 1e-9 under a large diagonal g: their own 53 bits, not 2^-60."""
    rng = np.random.default_rng(55)
    V = int(np.prod(DIMS))
    small = 1e-9 * (rng.normal(size=(4, V, 3, 3)) + 1j * rng.normal(size=(4, V, 3, 3)))
    U = (np.eye(3) * (1 - 1e-9j) + small - np.swapaxes(small, -1, -2).conj()).reshape((4,) + DIMS[::-1] + (3, 3))
    ph = rng.uniform(-3, 3, size=(V, 2))
    ph = np.exp(1j * np.concatenate([ph, -ph.sum(1, keepdims=True)], 1))
    g = (np.eye(3) * ph[:, None, :]).reshape(DIMS[::-1] + (3, 3))
    U, g = np.ascontiguousarray(U), np.ascontiguousarray(g)
    out, ref = update(U, g), expected(U, g)
    off = ~np.eye(3, dtype=bool)
    err = (np.abs(out - ref).astype(float))[..., off].max()
    assert err < 32 * 2.0 ** -53 * 1e-8, err
