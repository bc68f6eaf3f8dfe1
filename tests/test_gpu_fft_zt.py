"""The pass over z and t with the filter (k_fx_zt), in float and double-float, against the three column passes (LGF_FFT_ZT=0): the same
bits for every pair of extents that takes it and for the pairs beside its limit, and for a batch."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PAIRS = [(nz, nt) for nz in (8, 16, 24, 32, 48, 64) for nt in (8, 16, 24, 32, 48, 64)]


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nxy", [8, 24])
def test_same_bits_as_column_passes(nxy, precision, monkeypatch):
    import torch

    import paper_1210_8018_gb300 as lgf
    gen = torch.Generator(device="cuda").manual_seed(91)
    for nz, nt in PAIRS:
        d = torch.randn(nt, nz, nxy, nxy, 3, 3, dtype=torch.complex128, device="cuda", generator=gen)
        d = d - d.mH
        d = d - torch.diagonal(d, dim1=-2, dim2=-1).mean(-1)[..., None, None] * torch.eye(3, device="cuda")
        out = []
        for flag in ("1", "0"):
            monkeypatch.setenv("LGF_FFT_ZT", flag)
            with lgf.Lattice((nxy, nxy, nz, nt)) as lat:
                out.append(torch.empty_like(d))
                lat.filter(d, out[-1], precision)
        assert torch.equal(out[0], out[1]), (nz, nt)


def test_batch_mixed(monkeypatch):
    import paper_1210_8018_gb300 as lgf
    import synth
    dims = [(8, 8, 8, 16)] * 3 + [(8, 8, 24, 8)]
    res = []
    for flag in ("1", "0"):
        monkeypatch.setenv("LGF_FFT_ZT", flag)
        Us = [synth.config(d, 92 + k, 0.5) for k, d in enumerate(dims)]
        with lgf.Batch(dims) as b:
            r = b.fix(Us, 0.08, 1e-15, "mixed")
        assert all(x["theta"] < 1e-15 for x in r)
        res.append(Us)
    assert all(np.array_equal(a, b) for a, b in zip(*res))
