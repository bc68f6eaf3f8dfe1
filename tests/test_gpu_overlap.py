"""Outputs of the functional, its gradient and the update that lie over their inputs: the same bits as apart. The
lattice is large enough that blocks which start late would read what the first ones have written."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

DIMS = (24, 16, 16, 16)
SITES = int(np.prod(DIMS))


@pytest.fixture(scope="module")
def fields():
    import torch
    U = torch.from_numpy(synth.config(DIMS, 111, 0.6)).cuda()
    gen = torch.Generator(device="cuda").manual_seed(112)
    w = 0.3 * torch.randn(SITES, 8, dtype=torch.float64, device="cuda", generator=gen)
    w[5] *= 40  # by eigenvectors
    return U, w


def test_g_over_omega(fields):
    import torch
    import paper_1210_8018_gb300 as lgf
    U, w = fields
    g = torch.empty_like(U[0])
    buf = torch.empty_like(U[0])
    omega = torch.view_as_real(buf).reshape(-1)[:8 * SITES].reshape(SITES, 8)
    omega.copy_(w)
    with lgf.Lattice(DIMS) as lat:
        F = lat.functional(U, w, g)
        assert lat.functional(U, omega, buf) == F
    assert torch.equal(buf, g)


# at the start of a direction's links, across two of them, and over omega: shifted by a site, and itself
@pytest.mark.parametrize("where", ["links", "across", "shifted", "omega"])
def test_gradient_over_its_inputs(fields, where):
    import torch
    import paper_1210_8018_gb300 as lgf
    U, w = fields
    V, omega = U.clone(), w.clone()
    flat = torch.view_as_real(V).reshape(-1)
    if where in ("links", "across"):
        first = 18 * SITES * 2 - (4 * SITES if where == "across" else 0)
        grad = flat[first:first + 8 * SITES].reshape(SITES, 8)
    else:
        both = torch.empty(8 * (SITES + 1), dtype=torch.float64, device="cuda")
        omega = both[:8 * SITES].reshape(SITES, 8)
        omega.copy_(w)
        grad = both[8:].reshape(SITES, 8) if where == "shifted" else omega
    ref = torch.empty_like(w)
    with lgf.Lattice(DIMS) as lat:
        lat.functional_grad(U, w, ref)
        lat.functional_grad(V, omega, grad)
    assert torch.equal(grad, ref)


def test_update_by_its_own_links(fields):
    import torch
    import paper_1210_8018_gb300 as lgf
    U, _ = fields
    apart, over = U.clone(), U.clone()
    with lgf.Lattice(DIMS) as lat:
        lat.update(apart, U[2].contiguous())
        lat.update(over, over[2])
    assert torch.equal(apart, over)
