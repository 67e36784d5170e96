"""The passes of a training step around the network's GEMMs at ragged sizes
(below one 32-column group, off every tile edge, batches that are not whole
128-row tiles): the bias gradient is one sequential FP32 sum per column, the
loss and its gradient those of the rows, Adam's update the formula's, and both
BF16 weight copies follow the FP32 weights."""
import numpy as np
import pytest

from test_gpu_mlp import init_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(1, 1, 1, 64), (33, 31, 70, 192), (130, 96, 33, 320), (65, 257, 128, 128)])
def test_a_training_step_at_ragged_sizes(built_lib, cuda, dims):
    import torch
    import paper_2608_21150_gb300 as P
    I, H, O, B = dims
    rng = np.random.default_rng(B + H)
    net, other = P.MLP(I, H, O, max_batch=384), P.MLP(I, H, O, max_batch=B)
    p = init_params(rng, I, H, O)
    net.set_params(p)
    other.set_params(p)
    x = torch.from_numpy(rng.standard_normal((B, I)).astype(np.float32)).to(cuda)
    t = torch.from_numpy(rng.standard_normal((B, O)).astype(np.float32)).to(cuda)
    y = torch.empty((B, O), dtype=torch.float32, device=cuda)
    lr = 1e-2
    # forward, loss gradient and backward by hand
    other.forward(x, y)
    d = (y - t).cpu().numpy()
    dy = np.float32(2.0) / (np.float32(B) * np.float32(O)) * d
    other.backward(torch.from_numpy(dy).to(cuda))
    g = other.grads()
    seq = np.zeros(O, dtype=np.float32)
    for r in range(B):
        seq = seq + dy[r]
    assert np.array_equal(g[-O:], seq)
    # the same in one training step: B terms of FP64 per row and then over the rows
    loss = net.train_step(x, t, lr)
    assert abs(loss - np.mean(d.astype(np.float64) ** 2)) < 1e-13 * loss + 1e-300
    assert np.array_equal(net.grads(), g)
    # first Adam step: the bias corrections cancel (1 - beta); ten FP32 roundings of an update of at most lr
    other.adam(lr)
    w = other.params()
    assert np.array_equal(net.params(), w)
    g64 = g.astype(np.float64)
    ref = p - lr * g64 / (np.abs(g64) + 1e-8)
    assert np.all(np.abs(w - ref) <= 6e-8 * np.abs(ref) + 2e-6 * lr)
    # the BF16 copies that the next step's GEMMs read
    fresh = P.MLP(I, H, O, max_batch=B)
    fresh.set_params(w)
    y2 = torch.empty_like(y)
    net.forward(x, y)
    fresh.forward(x, y2)
    assert torch.equal(y, y2)
    for n in (net, fresh):
        n.backward(torch.from_numpy(dy).to(cuda))
    assert np.array_equal(net.grads(), fresh.grads())
