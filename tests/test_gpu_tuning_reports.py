"""The set-up timings that a model reports are those of what they name: the symmetric-state path's are measured beside the
loop launch shapes, for either products backend, and a second model of the shape reports the same ones."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1710_08830_gb300 import inputs  # noqa: E402


@pytest.mark.parametrize("products", ["SIMT", "TC"])
def test_symmetric_state_timings_are_reported(products):
    from paper_1710_08830_gb300 import api
    spec = inputs.rashba_hubbard(1.0, -0.2, 0.3, 2.5, -0.818, Lq=10, nc=8, n_ff=9)
    reports = []
    for _ in range(2):
        m = api.Model(spec, api.SPLIT32, products=getattr(api, "PRODUCTS_" + products))
        assert m.symmetric_state_path and len(m.loop_tiles_tuning_ms) > 1
        reports.append(m.symmetric_state_tuning_ms)
    assert reports[0] == reports[1] and all(v > 0 for v in reports[0].values())
