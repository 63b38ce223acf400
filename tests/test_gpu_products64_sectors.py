"""Entry-wise accuracy of the FP64 products of large matrices: every entry of c A L A is within the rounding bound of plain
FP64 sums of the same products, 2 M roundings per complex sum and product, however small it is beside the rest of its row
and column (blocks of very different size that the loops do not mix, entries over many orders of magnitude)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1710_08830_gb300 import inputs  # noqa: E402

U = 2.0 ** -53


def _loop_matrix(spec, deltas, Lc):
    """L[(R1,a),(R2,b)] of one momentum from its compact loops."""
    b = [tuple(int(x) for x in v) for v in spec.ff_R]
    at = {tuple(int(x) for x in v): i for i, v in enumerate(deltas)}
    n2 = spec.n_s ** 2
    L = np.empty((spec.n_ff, n2, spec.n_ff, n2), complex)
    for i, p in enumerate(b):
        for j, q in enumerate(b):
            L[i, :, j, :] = Lc[at[(p[0] - q[0], p[1] - q[1])]]
    return L.reshape(spec.M, spec.M)


def _check(m, spec, X, mask, ch, T=0.4):
    """One channel's products at a sample of rows of one momentum against extended precision."""
    A = m.project(X, mask=mask)[0].cpu().numpy()[ch]
    Lc = m.loops(T, mask=mask).cpu().numpy()[ch]
    d = m.rhs(T, X, mask=mask).cpu().numpy()[ch]
    rows = np.linspace(0, spec.M - 1, 8).astype(int)
    for q in (spec.Nq - 1,):
        L = _loop_matrix(spec, m.deltas, Lc[q])
        a, l = A[q].astype(np.clongdouble), L.astype(np.clongdouble)
        exact = (1 + ch) * (a[rows] @ l) @ a
        size = (1 + ch) * (np.abs(A[q][rows]) @ np.abs(L)) @ np.abs(A[q])
        # per product and part 2 M roundings of sums of complex terms, both parts: 2 sqrt(2) M u; two products, and the scale
        bound = (4 * np.sqrt(2.0) * spec.M + 8) * U * size
        assert (np.abs((d[q][rows] - exact).astype(complex)) <= bound).all()


def _decoupled():
    """Four orbitals that nothing couples: the loops are diagonal in the orbital pairs."""
    s = inputs.rashba_bilayer(Lq=3, nc=2, n_ff=9)
    t = np.array([np.diag(np.diag(x).real * (1 + 0.1 * np.arange(4))) for x in s.hop_t]).astype(complex)
    return s.with_(hop_t=t, V0=np.zeros_like(s.V0))


def _block_state(spec, eps, seed=1):
    """P of two blocks of orbital pairs, rows of the first with small entries towards the second (0 the other way)."""
    r = np.random.default_rng(seed)
    X = np.zeros((2, spec.Nq, spec.M, spec.M), complex)
    second = (np.arange(spec.M) % spec.n_s ** 2) % 2 == 1
    scale = np.where(second[None, :], np.where(second[:, None], 1.0, eps), np.where(second[:, None], 0.0, 1.0))
    X[0] = (r.standard_normal(X[0].shape) + 1j * r.standard_normal(X[0].shape)) * scale
    return X


@pytest.mark.parametrize("eps", [1.0, 1e-3, 1e-9, 1e-30])
def test_blocks_of_different_size(eps):
    from paper_1710_08830_gb300 import api
    spec = _decoupled()
    m = api.Model(spec, api.FP64)
    _check(m, spec, _block_state(spec, eps), api.CH_P, 0)


@pytest.mark.parametrize("model,n_ff,Lq", [("bilayer", 5, 3), ("bilayer", 9, 3), ("t2g", 5, 3), ("bilayer", 13, 5), ("t2g", 9, 3)])
def test_entries_over_many_orders(model, n_ff, Lq):
    from paper_1710_08830_gb300 import api
    spec = (inputs.t2g_soc(1, 0.2, 2.0, 0.4, Lq=Lq, nc=1, n_ff=n_ff).with_(mu=0.1, filling=0.0) if model == "t2g" else
            inputs.rashba_bilayer(Lq=Lq, nc=1, n_ff=n_ff))
    m = api.Model(spec, api.FP64)
    st = inputs.random_state(spec, seed=2, scale=0.3)
    wide = st * np.exp(np.random.default_rng(4).uniform(-25, 3, st.shape))
    sparse = wide * (np.random.default_rng(5).random(st.shape) < 0.03)
    for X in (st, wide, sparse):
        for mask, ch in ((api.CH_P, 0), (api.CH_C, 1)):
            _check(m, spec, X, mask, ch)


@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_not_finite_where_a_sum_is_not(bad):
    from paper_1710_08830_gb300 import api
    spec = _decoupled()
    m = api.Model(spec, api.FP64)
    X = _block_state(spec, 1e-9)
    X[0, 4, 6, 20] = bad
    d = np.isfinite(m.rhs(0.4, X, mask=api.CH_P).cpu().numpy()[0, 4])
    # T = A L: row 6; T A: row 6, and column 20 (a zero times an infinity is not finite either)
    want = np.ones((spec.M, spec.M), bool)
    want[6, :] = False
    want[:, 20] = False
    assert np.array_equal(d, want)
