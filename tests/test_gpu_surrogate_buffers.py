"""A network's buffers move when a larger batch passes through it: flows that hold its captured evaluations are captured again,
and models that share a network in a batch of flows take turns on its buffers."""
import ctypes as C
from types import SimpleNamespace

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1710_08830_gb300 import inputs  # noqa: E402


def _net():
    from paper_1710_08830_gb300.surrogate import Net
    n_out = 2 * 25 * 16 * 2
    net = Net(20, 64, 2, n_out, seed=3)
    # small loops from an untrained network, never refused: what counts is that its evaluations are the same
    return SimpleNamespace(net=net, mean=np.zeros(n_out, np.float32), std=np.full(n_out, 1e-3, np.float32))


def _model(tr, Lq, tp=-0.2, stream=None):
    from paper_1710_08830_gb300 import api
    from paper_1710_08830_gb300.surrogate import attach
    m = api.Model(inputs.rashba_hubbard(tp=tp, alpha=0.3, U=2.5, mu=-0.8, Lq=Lq, nc=2, n_ff=9), api.SPLIT32, stream=stream)
    attach(m, tr, 0.3, tp, -0.8, tol=1e30, n_check=4)
    return m


def _grow(tr, batch):
    X, Y = torch.zeros((batch, 20), device="cuda"), torch.zeros((batch, tr.net.n_out), device="cuda")
    tr.net.gradients(X, Y)


FLOW = dict(T0=1.0, T_end=0.3, rtol=1e-3, atol=1e-3, h0=-0.2)
KEYS = ("n_steps", "n_reject", "n_rhs", "amax", "T_last")


def test_flow_after_the_network_has_grown():
    tr = _net()
    m = _model(tr, 6)
    X, r = m.flow(**FLOW)
    assert r["n_rhs"] > 6
    _grow(tr, 1000)
    Y, s = m.flow(**FLOW)
    assert torch.equal(X, Y) and all(r[k] == s[k] for k in KEYS)


def test_stepwise_flow_while_the_network_grows():
    from paper_1710_08830_gb300._lib import FlowOpts, FlowResult, FlowStepInfo
    tr = _net()
    m = _model(tr, 6)
    X, r = m.flow(**FLOW)
    o = FlowOpts(FLOW["T0"], FLOW["T_end"], FLOW["rtol"], FLOW["atol"], FLOW["h0"], 50.0, 3, 1000)
    info, res, Y = FlowStepInfo(), FlowResult(), m.zeros_state()
    m._check(m._L.tufrg_flow_start(m._h, C.byref(o)))
    for i in range(1000):
        m._check(m._L.tufrg_flow_step(m._h, C.byref(info)))
        if info.status != 0:
            break
        _grow(tr, 300 * (i + 1))
    m._check(m._L.tufrg_flow_end(m._h, C.c_void_p(Y.data_ptr()), C.byref(res)))
    assert torch.equal(X, Y) and res.n_steps == r["n_steps"]


def test_batched_flows_that_share_a_network():
    from paper_1710_08830_gb300 import api
    args = [(4, -0.2), (6, -0.1), (8, -0.25)]   # each grows the network for the one before
    single = [_model(_net(), Lq, tp).flow(**FLOW)[1] for Lq, tp in args]
    tr = _net()
    batch = api.flow_batch([_model(tr, Lq, tp, torch.cuda.Stream()) for Lq, tp in args], **FLOW)
    for a, b in zip(single, batch):
        assert all(a[k] == b[k] for k in KEYS)
