"""The kernels of an iteration launched behind one another (LGF_PDL) against ordinary launches: the same bits from
every schedule and from a batch's graph, on lattices whose kernels are short and on one with several waves of blocks,
by the fixed-length and the general FFT passes."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("dims", [(8, 8, 8, 8), (10, 9, 8, 6), (24, 24, 24, 32)])
def test_same_bits(dims, precision, monkeypatch):
    import torch
    import paper_1210_8018_gb300 as lgf
    U = torch.from_numpy(synth.config(dims, 131, 0.5)).cuda()
    runs = []
    for flag in ("1", "0"):
        monkeypatch.setenv("LGF_PDL", flag)
        V = U.clone()
        with lgf.Lattice(dims) as lat:
            r = lat.fix(V, 0.08, 1e-15, precision)
        assert r["theta"] < 1e-15
        runs.append((V, r["iters"], r["theta"], r["F"]))
    assert torch.equal(runs[0][0], runs[1][0]) and runs[0][1:] == runs[1][1:]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_same_bits_in_a_batch(precision, monkeypatch):
    import paper_1210_8018_gb300 as lgf
    monkeypatch.setenv("LGF_AUTOTUNE", "0")
    dims = [(8, 8, 8, 8), (10, 9, 8, 6), (8, 8, 8, 8)]
    runs = []
    for flag in ("1", "0"):
        monkeypatch.setenv("LGF_PDL", flag)
        Us = [synth.config(d, 132 + k, 0.5) for k, d in enumerate(dims)]
        with lgf.Batch(dims) as b:
            r = b.fix(Us, 0.08, 1e-15, precision)
        runs.append((Us, r))
    assert all(np.array_equal(a, b) for a, b in zip(runs[0][0], runs[1][0])) and runs[0][1] == runs[1][1]
