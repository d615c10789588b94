"""The network's tensor-core passes (fused forward and backward data on padded
planes, weight gradients by slabs) against the FP64 oracle at the shapes where
their tiling can go wrong: boxes of one voxel, one row or one slice, one row
tile and several, widths that are no multiple of anything, hidden widths below,
at and between the padded 16 and 32, one sample and more samples than SMs, two
layers (no hidden convolution), more than eight input channels (per-layer
kernels) and a box whose planes do not fit shared memory (likewise).

Tolerances: a layer sums at most 32 x 27 products in FP32, whose rounding is at
most about sqrt(864) 2^-24 = 1.8e-6 of the sum of magnitudes; the forward bound
is that of the other learned tests, the gradient's the FP32 bar 2e-5."""
import numpy as np
import pytest

from oracle import conv3d

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# D, H, W, in, hidden, layers, batch
CASES = [(1, 1, 1, 4, 8, 2, 1), (1, 1, 7, 4, 16, 3, 2), (1, 9, 1, 2, 32, 3, 3), (3, 1, 1, 8, 12, 4, 1),
         (2, 3, 5, 4, 24, 3, 5), (5, 10, 10, 4, 32, 4, 3), (3, 9, 8, 4, 16, 5, 4), (8, 4, 4, 1, 32, 4, 2),
         (4, 5, 6, 4, 8, 3, 200), (5, 10, 10, 9, 32, 3, 2), (8, 10, 10, 4, 32, 4, 2)]


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("weighted", [False, True])
def test_passes_match_the_oracle(case, weighted):
    from paper_2103_08513_gb300.learned import WarmStartNet
    D, H, W, cin0, hidden, layers, batch = case
    net = WarmStartNet(D, H, W, hidden=hidden, layers=layers, in_channels=cin0, batch=batch, seed=3)
    gen = torch.Generator().manual_seed(11)
    cin = [cin0] + [hidden] * (layers - 1)
    cout = [hidden] * (layers - 1) + [1]
    off = 0
    for ci, co in zip(cin, cout):                       # non-zero biases
        off += co * ci * 27
        net.master[off:off + co] = (0.1 * torch.randn(co, generator=gen)).cuda()
        off += co
    net.sync_weights()
    x = torch.randn((batch, cin0, D, H, W), generator=gen)
    t = torch.rand((batch, 1, D, H, W), generator=gen)
    w = torch.rand((batch, 1, D, H, W), generator=gen) if weighted else None
    y = net.forward(x.cuda())
    grad, loss = net.gradient(x.cuda(), t.cuda(), weight=None if w is None else w.cuda())
    torch.cuda.synchronize()
    flat = net.bf16_weights().cpu().numpy().astype(np.float64)
    master = net.master.cpu().numpy().astype(np.float64)
    off = 0
    for ci, co in zip(cin, cout):
        off += co * ci * 27
        flat[off:off + co] = master[off:off + co]
        off += co
    params = conv3d.unflatten(flat, cin, cout)
    xd, td = x.numpy().astype(np.float64), t.numpy().astype(np.float64)
    yr = conv3d.forward(params, xd)[-1]
    assert np.abs(y.cpu().numpy() - yr).max() <= 2e-6
    lref, gref = conv3d.loss_and_grad(params, xd, td, None if w is None else w.numpy().astype(np.float64))
    gref = conv3d.flatten(gref)
    g = grad.cpu().numpy()
    print(case, "forward", np.abs(y.cpu().numpy() - yr).max(), "gradient", np.linalg.norm(g - gref) / np.linalg.norm(gref))
    assert abs(float(loss.cpu()[0]) - lref) <= 1e-5 * lref
    assert np.linalg.norm(g - gref) <= 2e-5 * np.linalg.norm(gref)
