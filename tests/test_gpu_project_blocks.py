"""The multi-orbital split projections (whole orbital blocks staged per bond pair) against the FP64 per-entry kernel, at one
and several bond pairs, momentum lists that do not fill a group, single channels, and lists of orbit representatives."""
import numpy as np
import pytest

from paper_1710_08830_gb300 import inputs

pytestmark = pytest.mark.gpu


# the split path projects an FP32 rounding of the state: every sum has at most 2 n_ff + 1 terms of rounded factors
@pytest.mark.parametrize("make", [inputs.rashba_bilayer, inputs.t2g_soc])
@pytest.mark.parametrize("Lq,nc,n_ff", [(2, 2, 1), (3, 2, 5), (5, 1, 9), (12, 1, 5)])
@pytest.mark.parametrize("mask", [1, 2, 3])
def test_block_projections_match_fp64(make, Lq, nc, n_ff, mask):
    from paper_1710_08830_gb300 import api
    spec = make(Lq=Lq, nc=nc, n_ff=n_ff)
    X = inputs.random_state(spec, 5)
    ref, mref = api.Model(spec, api.FP64).project(X, mask=mask)
    A, mx = api.Model(spec, api.SPLIT32).project(X, mask=mask)
    ref, A = ref.cpu().numpy(), A.cpu().numpy()
    for ch in range(2):
        if mask >> ch & 1:
            assert np.abs(A[ch] - ref[ch]).max() <= 2e-6 * np.abs(ref).max()
    assert abs(mx - mref) <= 2e-6 * mref


@pytest.mark.parametrize("make", [inputs.rashba_bilayer, inputs.t2g_soc])
def test_products_into_an_output_off_the_32_byte_grid(make):
    """16-byte aligned outputs take two stores per pair of entries instead of one and hold the same bits"""
    import torch

    from paper_1710_08830_gb300 import api
    spec = make(Lq=3, nc=2, n_ff=5)
    m = api.Model(spec, api.SPLIT32, products=api.PRODUCTS_TC)
    X = m._dev(inputs.random_state(spec, 3))
    a = m.rhs(0.4, X).clone()
    buf = torch.empty(X.numel() + 1, dtype=torch.complex128, device=X.device)
    out = buf[1:].view(X.shape)
    assert out.data_ptr() % 32 == 16
    b = m.rhs(0.4, X, out=out)
    assert torch.equal(a, b)
