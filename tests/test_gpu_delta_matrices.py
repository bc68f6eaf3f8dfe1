"""Delta from the caller's links to the caller's matrices in one pass (k_delta_matrices): ragged last warps and
blocks, several sites per thread, host and device memory, and an output that lies over the links."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (3, 5, 3, 5), (9, 4, 8, 8), (16, 16, 16, 18)])
@pytest.mark.parametrize("where", ["device", "host", "over"])
def test_delta_matrices(dims, where):
    import torch

    import paper_1210_8018_gb300 as lgf
    U = synth.config(dims, 81, 0.6)
    ref = oracle.delta(U)
    with lgf.Lattice(dims) as lat:
        if where == "host":
            out = np.empty_like(ref)
            theta, F = lat.delta(U, out)
        else:
            Ud = torch.from_numpy(U.copy()).cuda()
            D = Ud[2] if where == "over" else torch.empty_like(Ud[0])
            theta, F = lat.delta(Ud, D)
            out = D.cpu().numpy()
    # sixteen terms of magnitude below 1, summed in double on one side, in fixed point on the other
    assert np.abs(out - ref).max() < 16 * 2.0 ** -52
    assert abs(theta - (np.abs(ref) ** 2).sum() / (3 * ref[..., 0, 0].size)) < 1e-13 * theta
    assert abs(F - np.trace(U, axis1=-2, axis2=-1).real.mean() / 3) < 1e-13
    assert np.array_equal(out[..., 1, 0], -out[..., 0, 1].conj()) and not out[..., 0, 0].real.any()
