"""The network's passes at the shapes where tiles, stages, packed chunks and partial sums are ragged: batches around the
128-row tiles and the partial sums' rows, widths that are not multiples of 4 (no vector accesses), 8 or 16, one to five
layers, and a smaller batch after a larger one (the operand scratch is kept).  Gradients against the FP64 network within
the BF16 rounding bound of the training pass, inference within FP32 accuracy."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import mlp  # noqa: E402

SHAPES = [(20, 256, 4, 1600, (1024, 1000, 129)), (7, 33, 1, 5, (1, 8, 9, 127)), (3, 100, 2, 513, (128, 17)), (20, 64, 3, 2, (2049, 64))]


@pytest.mark.parametrize("n_in,width,depth,n_out,batches", SHAPES)
def test_passes_at_ragged_shapes(n_in, width, depth, n_out, batches):
    from paper_1710_08830_gb300.surrogate import Net
    rng = np.random.default_rng(5)
    net = Net(n_in, width, depth, n_out, seed=3)
    shapes = mlp.layer_shapes(n_in, width, depth, n_out)
    p = net.get_params()
    p += rng.normal(0, 0.05, p.size).astype(np.float32)      # biases that are not zero
    net.set_params(p)
    pw = p.astype(np.float64)                                # the weights the kernels use: rounded to BF16
    o = 0
    for din, dout in shapes:
        w = torch.from_numpy(p[o:o + din * dout]).to(torch.bfloat16).double().numpy()
        pw[o:o + din * dout] = w
        o += din * dout + dout
    for b in batches:
        X = rng.uniform(-1, 1, (b, n_in)).astype(np.float32)
        T = rng.normal(0, 1, (b, n_out)).astype(np.float32)
        Xd, Td = torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda()
        loss, g = net.gradients(Xd, Td)
        ref_loss, ref = mlp.loss_and_grad(pw, shapes, X, T)
        assert abs(loss - ref_loss) <= 2 * (depth + 1) * 2.0 ** -8 * ref_loss
        assert np.linalg.norm(g.cpu().numpy() - ref) <= 2 * (depth + 1) * 2.0 ** -8 * np.linalg.norm(ref)
        Y, _ = mlp.forward(pw, shapes, X)
        assert np.linalg.norm(net.forward(Xd).cpu().numpy() - Y) <= 1e-5 * np.linalg.norm(Y)
    net.close()
