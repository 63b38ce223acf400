"""A batch whose buffers do not fit is refused with TUFRG_ENOMEM and leaves the network usable: the next smaller batch gets
buffers of its own again."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MIB = 1 << 20


def test_network_after_a_batch_that_does_not_fit():
    from paper_1710_08830_gb300 import api
    from paper_1710_08830_gb300.surrogate import Net
    net = Net(20, 64, 2, 400)
    r = np.random.default_rng(3)
    X = torch.from_numpy(r.standard_normal((131072, 20)).astype(np.float32)).cuda()
    Y = torch.from_numpy(r.standard_normal((131072, 400)).astype(np.float32)).cuda()   # 200 MiB
    loss, g = net.gradients(X[:64].contiguous(), Y[:64].contiguous())
    small = (X[:64].contiguous(), Y[:64].contiguous())
    torch.cuda.synchronize()
    free, _ = torch.cuda.mem_get_info()
    # 131072 rows need 200 MiB of outputs and twice as much of upstream gradients
    blocker = torch.empty((free - 256 * MIB) // (2 * MIB) * (2 * MIB), dtype=torch.uint8, device="cuda")
    try:
        with pytest.raises(api.TufrgError) as e:
            net.gradients(X, Y)
        assert e.value.status == 2, e.value
    finally:
        del blocker
        torch.cuda.empty_cache()
    loss2, g2 = net.gradients(*small)
    assert loss2 == loss and torch.equal(g2, g)
