"""FP64 products of large matrices from integer digits on the tensor cores, through one right-hand side, against the
oracle: orders around the 128-row and 32-column tiles, the 16-value stages and the 256-value exact sums (M = 80, 144, 180,
208, 324), states whose entries span many orders of magnitude, single channels, and states with entries that are not
finite (the affected products are not finite, the others are untouched)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_1710_08830_gb300 import inputs  # noqa: E402


def _spec(model, n_ff, Lq):
    if model == "t2g":
        return inputs.t2g_soc(1, 0.2, 2.0, 0.4, Lq=Lq, nc=1, n_ff=n_ff).with_(mu=0.1, filling=0.0)
    return inputs.rashba_bilayer(Lq=Lq, nc=1, n_ff=n_ff)


def rel(a, b):
    return np.abs(a - b).max() / np.abs(b).max()


@pytest.mark.parametrize("model,n_ff,Lq", [("bilayer", 5, 3), ("bilayer", 9, 3), ("t2g", 5, 3), ("bilayer", 13, 5), ("t2g", 9, 3)])
def test_products_match_oracle(model, n_ff, Lq):
    from paper_1710_08830_gb300 import api
    spec = _spec(model, n_ff, Lq)
    m = api.Model(spec, api.FP64)
    o = oracle.Oracle(spec)
    st = inputs.random_state(spec, seed=2, scale=0.3)
    wide = st * np.exp(np.random.default_rng(4).uniform(-25, 3, st.shape))   # no symmetry, 1e-11 .. 20
    for X in (st, wide):
        ref, _ = o.rhs(0.4, X, 3)
        assert rel(m.rhs(0.4, X).cpu().numpy(), ref) < 1e-12
        for mask, ch in ((api.CH_P, 0), (api.CH_C, 1)):
            one, _ = o.rhs(0.4, X, mask)
            d = m.rhs(0.4, X, mask=mask).cpu().numpy()
            assert rel(d[ch], one[ch]) < 1e-12 and not np.any(d[1 - ch])


def test_products_of_states_that_are_not_finite():
    """An entry X_P(q) that is not finite reaches the P products of q (and, through the bond transforms, the C products)."""
    from paper_1710_08830_gb300 import api
    spec = _spec("bilayer", 5, 3)
    m = api.Model(spec, api.FP64)
    st = inputs.random_state(spec, seed=2, scale=0.3)
    good = m.rhs(0.4, st, mask=api.CH_P).cpu().numpy()
    for bad in (np.nan, np.inf):
        X = st.copy()
        X[0, 4, 7, 11] = bad
        d = m.rhs(0.4, X, mask=api.CH_P).cpu().numpy()   # P alone: momenta do not mix
        assert not np.isfinite(d[0, 4]).all()
        others = [q for q in range(9) if q != 4]
        assert np.array_equal(d[0, others], good[0, others])
