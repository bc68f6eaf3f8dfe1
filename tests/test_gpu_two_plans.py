"""Two lattices alive at the same time whose plans ask different amounts of shared memory of the same kernel: the
general FFT pass (110 KB for z and t of 24 x 36 in float, 51 KB for 20 x 20; both above the 48 KB that need no
opting in)."""
import pytest

import oracle

pytestmark = pytest.mark.gpu

LARGE, SMALL = (30, 20, 24, 36), (20, 20, 20, 20)


def test_larger_plan_after_a_smaller_one():
    import torch
    import paper_1210_8018_gb300 as lgf
    gen = torch.Generator(device="cuda").manual_seed(5)
    c = torch.randn(LARGE[::-1] + (8,), dtype=torch.float64, device="cuda", generator=gen)
    d = torch.randn(SMALL[::-1] + (8,), dtype=torch.float64, device="cuda", generator=gen)
    out = [torch.empty_like(c), torch.empty_like(d), torch.empty_like(c)]
    with lgf.Lattice(LARGE) as a, lgf.Lattice(SMALL) as b:
        a.filter_coeffs(c, out[0], "fp32")
        b.filter_coeffs(d, out[1], "fp32")
        a.filter_coeffs(c, out[2], "fp32")
    assert torch.equal(out[0], out[2]) and bool(torch.isfinite(out[1]).all())


def test_batch_of_both(monkeypatch):
    import paper_1210_8018_gb300 as lgf
    import synth
    monkeypatch.setenv("LGF_AUTOTUNE", "0")
    dims = [LARGE, SMALL, SMALL]
    Us = [synth.config(d, 95 + k, 0.3) for k, d in enumerate(dims)]
    before = [oracle.plaquette(U) for U in Us]
    with lgf.Batch(dims) as b:
        r = b.fix(Us, 0.08, 1e-12, "mixed")
    assert all(x["theta"] < 1e-12 for x in r)
    for U, p in zip(Us, before):
        assert oracle.theta(oracle.delta(U)) < 1e-12 * (1 + 1e-6)
        assert abs(oracle.plaquette(U) - p) < 1e-14
