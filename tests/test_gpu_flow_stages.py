"""One attempt of the device flow (loops of the stages running ahead on the second stream, the last two stages sharing
theirs) against the Dormand-Prince step formed on the host from six evaluations of the right-hand side."""
import numpy as np
import pytest

from paper_1710_08830_gb300 import inputs

pytestmark = pytest.mark.gpu

C = [0, 1 / 5, 3 / 10, 4 / 5, 8 / 9, 1, 1]
A = [[], [1 / 5], [3 / 40, 9 / 40], [44 / 45, -56 / 15, 32 / 9],
     [19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729],
     [9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656],
     [35 / 384, 0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84]]


def _spec(name):
    if name == "two_band":
        return inputs.rashba_hubbard(1.0, -0.2, 0.3, 2.5, -0.7, Lq=5, nc=3, n_ff=9)
    if name == "two_band_one":   # a single transfer momentum and form factor
        return inputs.rashba_hubbard(1.0, -0.2, 0.3, 2.5, -0.7, Lq=2, nc=1, n_ff=1)
    if name == "shell":
        return inputs.rashba_hubbard(1.0, -0.2, 0.3, 2.5, -0.7, Lq=4, nc=2, n_ff=5).with_(regulator=1, T_reg=0.1)
    return {"bilayer": inputs.rashba_bilayer, "t2g": inputs.t2g_soc}[name](Lq=3, nc=2, n_ff=5)


# the split evaluations agree with FP64 to 2e-5 of the largest entry; the step is a sum of six of them with weights whose
# magnitudes add up to below 10 (their products with the stage errors enter at order h)
@pytest.mark.parametrize("prec,tol", [("FP64", 1e-9), ("SPLIT32", 2e-4)])
@pytest.mark.parametrize("name", ["two_band", "two_band_one", "shell", "bilayer", "t2g"])
@pytest.mark.parametrize("mask", [1, 2, 3])
@pytest.mark.parametrize("symmetric", [True, False])
def test_attempt_is_the_dormand_prince_step(name, mask, symmetric, prec, tol):
    from paper_1710_08830_gb300 import api
    m = api.Model(_spec(name), getattr(api, prec), symmetry=api.SYMMETRY_AUTO if symmetric else api.SYMMETRY_OFF)
    T0, h = 1.3, -0.05
    X, r = m.flow(T0=T0, T_end=T0 * float(np.exp(h)), rtol=1e3, atol=1e3, h0=2 * h, stop=1e6, mask=mask)
    assert r["n_steps"] == 1 and r["n_reject"] == 0
    k, y = [], np.zeros(X.shape, complex)
    for j in range(6):
        T = float(np.exp(np.log(T0) + C[j] * h))
        z = y + h * sum((a * v for a, v in zip(A[j], k)), np.zeros_like(y))
        k.append(T * m.rhs(T, m._dev(z), mask=mask).cpu().numpy())
    ref = y + h * sum(a * v for a, v in zip(A[6], k))
    assert np.abs(X.cpu().numpy() - ref).max() <= tol * np.abs(ref).max()


@pytest.mark.parametrize("prec", ["FP64", "SPLIT32"])
@pytest.mark.parametrize("name", ["two_band", "bilayer"])
def test_device_loop_is_the_flow_step_by_step(name, prec, tmp_path):
    """the loop on the device and single attempts on the host's call end in the same state, counts and step limit"""
    from paper_1710_08830_gb300 import api
    from paper_1710_08830_gb300._lib import TufrgError
    m = api.Model(_spec(name), getattr(api, prec))
    args = dict(T0=1.0, T_end=0.3, rtol=1e-3, atol=1e-3, h0=-0.2)
    X, r = m.flow(**args)
    Y, s = m.flow(**args, metrics_path=str(tmp_path / "m.jsonl"))
    assert (X == Y).all()
    for key in ("n_steps", "n_reject", "n_rhs", "amax", "T_last", "Tc", "crossed", "lead_channel", "lead_q"):
        assert r[key] == s[key], key
    with pytest.raises(TufrgError):
        m.flow(**args, max_steps=r["n_steps"] + r["n_reject"] - 1)
    Z, _ = m.flow(**args)
    assert (X == Z).all()
