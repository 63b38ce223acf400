"""The multi-orbital loops of the split path add the k-sum's FP32 accumulators (k_x ranges, real components, exchanged half,
1/Nk) in more than FP32, so ``loops`` returns values that FP32 cannot hold, at the representatives and at the momenta gathered
from them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1710_08830_gb300 import inputs  # noqa: E402


# several ranges of columns per momentum (few momenta), one range (tensor cores), every momentum summed
@pytest.mark.parametrize("model,Lq,nc,loops,symmetry", [
    ("bilayer", 12, 5, "AUTO", "AUTO"), ("bilayer", 5, 3, "AUTO", "OFF"), ("t2g", 5, 3, "SIMT", "AUTO"), ("t2g", 5, 3, "TC", "AUTO")])
def test_split_loops_hold_fp64_sums(model, Lq, nc, loops, symmetry):
    from paper_1710_08830_gb300 import api
    spec = (inputs.rashba_bilayer(Lq=Lq, nc=nc, n_ff=5) if model == "bilayer" else
            inputs.t2g_soc(1, 0.2, 2.0, 0.4, Lq=Lq, nc=nc, n_ff=5).with_(mu=0.1, filling=0.0))
    m = api.Model(spec, api.SPLIT32, loops=getattr(api, "LOOPS_" + loops), symmetry=getattr(api, "SYMMETRY_" + symmetry))
    L = m.loops(0.2)
    v = torch.view_as_real(L).reshape(2, spec.Nq, -1)
    beyond = (v != v.float().double()).sum(2)
    # (parts that vanish by symmetry apart; sums of few bits can be divisible by Nk = 225 or 3600, and then come many times)
    nonzero = (v != 0).sum(2)
    assert (nonzero > 0).all() and (beyond.double() / nonzero > 0.5).all()
    # and they agree with the FP64 model as FP32 k-sums do (the tolerance of the other comparisons of these loops)
    ref = api.Model(spec, api.FP64, symmetry=getattr(api, "SYMMETRY_" + symmetry)).loops(0.2)
    assert float((L - ref).abs().max() / ref.abs().max()) < 2e-5
