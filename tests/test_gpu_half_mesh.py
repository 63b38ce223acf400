"""The two-band k-sum over half of the fine mesh (exchange of the two propagators) against the oracle's sum over all of it,
at the shapes where the halves differ: odd and even fine meshes, transfer momenta with and without self-paired rows,
a second block of columns with one column, the smallest meshes, one to five y differences (FP64 splits the last two),
models with an inverting symmetry (both channels halved) and without (P only)."""
import numpy as np
import pytest

import oracle
from paper_1710_08830_gb300 import inputs

pytestmark = pytest.mark.gpu

# Lq, nc, n_ff: Lf = 15 (odd), 12 with odd cell (odd transfer momenta), 24, 65 (64 + 1 columns), 3, 2, 5, 18
SHAPES = [(5, 3, 9), (4, 3, 5), (6, 4, 13), (13, 5, 5), (3, 1, 9), (2, 1, 1), (5, 1, 13), (6, 3, 1)]


def rel(a, b):
    return np.abs(a - b).max() / max(1e-300, np.abs(b).max())


@pytest.mark.parametrize("prec,tol", [("FP64", 1e-10), ("SPLIT32", 2e-5)])
@pytest.mark.parametrize("Lq,nc,n_ff", SHAPES)
@pytest.mark.parametrize("variant", ["symmetric", "off", "shell", "no_inversion"])
def test_half_mesh_loops_match_oracle(Lq, nc, n_ff, prec, tol, variant):
    from paper_1710_08830_gb300 import api
    spec = inputs.rashba_hubbard(1.0, -0.2, 0.3, 2.5, -0.7, Lq=Lq, nc=nc, n_ff=n_ff)
    if variant == "shell":
        spec = spec.with_(regulator=1, T_reg=0.1)
    if variant == "no_inversion":   # a uniform bond current along x and a field: no symmetry inverts the momentum
        R, t = spec.hop_R.copy(), spec.hop_t.copy()
        for i, r in enumerate(R):
            if tuple(r) in ((1, 0), (-1, 0)):
                t[i] = t[i] + 0.15j * r[0] * np.eye(2) + 0.1j * r[0] * inputs.SIGMA_Z
        R = np.concatenate([R, [[0, 0]]]).astype(np.int32)
        t = np.concatenate([t, [0.2 * inputs.SIGMA_Z + 0.1 * inputs.SIGMA_X]])
        spec = spec.with_(hop_R=R, hop_t=t)
    m = api.Model(spec, getattr(api, prec), symmetry=api.SYMMETRY_OFF if variant == "off" else api.SYMMETRY_AUTO)
    o = oracle.Oracle(spec)
    L = m.loops(0.3).cpu().numpy()
    for ch, mask in ((0, api.CH_P), (1, api.CH_C)):
        ref = o.loops(0.3, ch)
        assert rel(L[ch], ref) < tol
        assert rel(m.loops(0.3, mask).cpu().numpy()[ch], ref) < tol


def _without_inversion(spec):
    """The model with a bond current along x and a site potential that breaks time reversal."""
    R, t = spec.hop_R.copy(), spec.hop_t.copy()
    n = spec.n_s
    Z = np.kron(np.eye(n // 2), inputs.SIGMA_Z)
    for i, r in enumerate(R):
        if tuple(r) in ((1, 0), (-1, 0)):
            t[i] = t[i] + 0.15j * r[0] * np.diag(np.arange(n) - n / 2) + 0.1j * r[0] * Z
    R = np.concatenate([R, [[0, 0]]]).astype(np.int32) if not any(tuple(r) == (0, 0) for r in R) else R
    if len(R) > len(t):
        t = np.concatenate([t, np.zeros((1, n, n), complex)])
    i0 = [tuple(r) for r in R].index((0, 0))
    t[i0] = t[i0] + 0.2 * Z + 0.1 * np.kron(np.diag(np.arange(n // 2)), np.eye(2)) + 0.1 * np.kron(np.eye(n // 2), inputs.SIGMA_X)
    return spec.with_(hop_R=R, hop_t=t)


# (model, Lq, nc, n_ff, precision, loops backend): tensor cores (groups of three momenta, stages of four rows: ragged
# groups and rows, meshes below a stage), CUDA cores in both precisions, five y differences
MULTI = [("t2g", 5, 3, 9, "SPLIT32", "LOOPS_TC"), ("t2g", 4, 3, 5, "SPLIT32", "LOOPS_TC"), ("t2g", 3, 1, 9, "SPLIT32", "LOOPS_TC"),
         ("t2g", 2, 1, 1, "SPLIT32", "LOOPS_TC"), ("t2g", 6, 2, 1, "SPLIT32", "LOOPS_TC"), ("t2g", 4, 3, 5, "SPLIT32", "LOOPS_SIMT"),
         ("t2g", 5, 1, 13, "SPLIT32", "LOOPS_AUTO"), ("t2g", 3, 3, 5, "FP64", "LOOPS_AUTO"), ("t2g", 5, 1, 13, "FP64", "LOOPS_AUTO"),
         ("bilayer", 5, 3, 9, "SPLIT32", "LOOPS_AUTO"), ("bilayer", 4, 3, 5, "FP64", "LOOPS_AUTO"),
         ("bilayer", 6, 2, 13, "SPLIT32", "LOOPS_AUTO"), ("bilayer", 2, 1, 1, "FP64", "LOOPS_AUTO")]


@pytest.mark.parametrize("model,Lq,nc,n_ff,prec,loops", MULTI)
@pytest.mark.parametrize("variant", ["symmetric", "off", "shell", "no_inversion"])
def test_half_mesh_multi_orbital_loops_match_oracle(model, Lq, nc, n_ff, prec, loops, variant):
    from paper_1710_08830_gb300 import api
    kw = dict(Lq=Lq, nc=nc, n_ff=n_ff)
    spec = inputs.t2g_soc(1, 0.2, 2.0, 0.4, **kw) if model == "t2g" else inputs.rashba_bilayer(**kw)
    if variant == "shell":
        spec = spec.with_(regulator=1, T_reg=0.1)
    if variant == "no_inversion":
        spec = _without_inversion(spec)
    m = api.Model(spec, getattr(api, prec), symmetry=api.SYMMETRY_OFF if variant == "off" else api.SYMMETRY_AUTO, mu=0.15,
                  loops=getattr(api, loops))
    o = oracle.Oracle(spec.with_(mu=0.15, filling=0.0))
    L = m.loops(0.3).cpu().numpy()
    for ch, mask in ((0, api.CH_P), (1, api.CH_C)):
        ref = o.loops(0.3, ch)
        tol = 1e-10 if prec == "FP64" else 2e-5
        assert rel(L[ch], ref) < tol
        assert rel(m.loops(0.3, mask).cpu().numpy()[ch], ref) < tol
