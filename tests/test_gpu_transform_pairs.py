"""The FP64 transform's row pass (R_y and -R_y formed together) against the oracle's projections: meshes with and without a
row difference that is its own negative (even and odd Lq), differences that wrap, one to nine of them, single channels."""
import numpy as np
import pytest

import oracle
from paper_1710_08830_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lq,n_ff", [(2, 1), (3, 5), (4, 5), (4, 9), (5, 9), (6, 13), (9, 13)])
@pytest.mark.parametrize("mask", [1, 2, 3])
def test_fp64_projections_match_oracle(Lq, n_ff, mask):
    from paper_1710_08830_gb300 import api
    spec = inputs.rashba_hubbard(1.0, -0.2, 0.3, 2.5, -0.7, Lq=Lq, nc=1, n_ff=n_ff)
    X = inputs.random_state(spec, 7)
    A, mx = api.Model(spec, api.FP64).project(X, mask)
    ref, mref = oracle.Oracle(spec).project(X, mask)
    A = A.cpu().numpy()
    for ch in range(2):
        if mask >> ch & 1:
            assert np.abs(A[ch] - ref[ch]).max() <= 1e-13 * np.abs(ref).max()
    assert abs(mx - mref) <= 1e-13 * mref
