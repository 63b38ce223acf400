"""The FP64 products of large matrices take the scratch that fits: a model whose full scratch does not fit beside its other
buffers is set up with a smaller one, and its results are the same bits."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1710_08830_gb300 import inputs  # noqa: E402

MIB = 1 << 20


def test_scratch_shrinks_where_memory_is_short():
    from paper_1710_08830_gb300 import api
    spec = inputs.t2g_soc(1, 0.2, 2.0, 0.4, Lq=8, nc=1, n_ff=9).with_(mu=0.1, filling=0.0)
    X = torch.from_numpy(inputs.random_state(spec, seed=2, scale=0.3)).cuda()   # 205 MiB
    ref, out = torch.empty_like(X), torch.empty_like(X)
    api.Model(spec, api.FP64).close()   # (the library's own first allocations)
    torch.cuda.synchronize()
    free0, _ = torch.cuda.mem_get_info()
    m = api.Model(spec, api.FP64)
    m.rhs(0.4, X, out=ref)
    torch.cuda.synchronize()
    used = free0 - torch.cuda.mem_get_info()[0]
    m.close()
    # the digits of the 64 momenta alone are 64 x 9 MiB; the set-up needs a state (205 MiB) for a while
    assert used > 900 * MIB
    free, _ = torch.cuda.mem_get_info()
    blocker = torch.empty((free - (used - 200 * MIB)) // (2 * MIB) * (2 * MIB), dtype=torch.uint8, device="cuda")
    try:
        m = api.Model(spec, api.FP64)
        m.rhs(0.4, X, out=out)
        torch.cuda.synchronize()
        m.close()
    finally:
        del blocker
        torch.cuda.empty_cache()
    assert torch.equal(out, ref)
