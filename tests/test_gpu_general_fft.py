"""The FFT passes for general extents against numpy's transform, at the edges of their tiles: planes that do not
fill the last tile, columns that do not fill it, the x and y axes apart (planes beyond 96 KB), the z and t axes
together and apart (at and above the 112 KB limit), every radix, and the longest axis in each place."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

DIMS = [(2, 3, 2, 5), (10, 9, 25, 2), (25, 27, 5, 9), (6, 10, 30, 36), (4, 6, 32, 27), (4, 6, 40, 25), (128, 125, 2, 3),
        (1024, 2, 3, 2), (2, 1024, 2, 3), (3, 2, 1024, 2), (2, 3, 2, 1024), (81, 5, 3, 16)]


def filtered(c, dims):
    """p^2_max / p^2 on the Fourier transform of a field (Nt, Nz, Ny, Nx, ...), 0 at zero momentum."""
    p2, top = np.zeros(dims[::-1]), 0.0
    for ax, n in enumerate(dims[::-1]):
        p2 = p2 + (4 * np.sin(np.pi * np.arange(n) / n) ** 2).reshape([-1 if a == ax else 1 for a in range(4)])
        top += 4 * np.sin(np.pi * (n // 2) / n) ** 2
    p2[0, 0, 0, 0] = np.inf
    k = np.fft.fftn(c, axes=(0, 1, 2, 3)) * (top / p2)[..., None]
    return np.fft.ifftn(k, axes=(0, 1, 2, 3)).real


# double-float transforms err by about 2^-45 of the field's norm per axis, float ones by a few 2^-24 per stage
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 5e-6)])
@pytest.mark.parametrize("dims", DIMS)
def test_general_passes(dims, precision, tol):
    import torch
    import paper_1210_8018_gb300 as lgf
    rng = np.random.default_rng(sum(dims))
    c = rng.normal(size=dims[::-1] + (8,))
    ref = filtered(c, dims)
    with lgf.Lattice(dims) as lat:
        out = torch.empty(c.shape, dtype=torch.float64, device="cuda")
        lat.filter_coeffs(torch.from_numpy(c).to("cuda"), out, precision)
    err = np.abs(out.cpu().numpy() - ref).max()
    assert err <= tol * np.abs(ref).max(), err


def test_general_passes_in_ieee_double(monkeypatch):
    import torch
    import paper_1210_8018_gb300 as lgf
    monkeypatch.setenv("LGF_FFT_NATIVE_F64", "1")
    dims = (10, 9, 25, 6)
    c = np.random.default_rng(3).normal(size=dims[::-1] + (8,))
    ref = filtered(c, dims)
    with lgf.Lattice(dims) as lat:
        out = torch.empty(c.shape, dtype=torch.float64, device="cuda")
        lat.filter_coeffs(torch.from_numpy(c).to("cuda"), out)
    assert np.abs(out.cpu().numpy() - ref).max() <= 1e-13 * np.abs(ref).max()
