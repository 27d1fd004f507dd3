"""The surrogate network's work buffers as its batches grow."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1101_5803_gb300 import binding as b
    return b


@pytest.mark.parametrize("small", [64, 200])
def test_batch_that_does_not_fit_leaves_the_network_usable(binding, small):
    # more rows than any device has memory for: refused, and the calls that
    # follow (within and beyond the batch held before) are as without it
    x = torch.as_tensor(np.random.default_rng(1).standard_normal((small, 7)).astype(np.float32), device="cuda")
    t = torch.ones((small, 2), device="cuda")
    a, b = binding.MLP([7, 256, 256, 2], seed=3), binding.MLP([7, 256, 256, 2], seed=3)
    y0 = a.forward(x[:64])
    lib = binding.load_library()
    stream = torch.cuda.current_stream().cuda_stream
    rc = lib.mirage_mlp_forward(a.handle, x.data_ptr(), 2 ** 31 - 1, y0.data_ptr(), stream)
    assert rc == -3  # MIRAGE_ERR_NOMEM, before anything is launched
    y = torch.empty((small, 2), device="cuda")
    rc = lib.mirage_mlp_grad(a.handle, x.data_ptr(), t.data_ptr(), 2 ** 31 - 1, None, None, y.data_ptr(), stream)
    assert rc == -3
    assert torch.equal(a.forward(x[:64]), b.forward(x[:64]))
    assert torch.equal(a.forward(x), b.forward(x))
    for net in (a, b):
        net.train(x, t, 3, 32, 1e-3, seed=5)
        net.train_step(x, t, 1e-3)
    torch.cuda.synchronize()
    assert np.array_equal(a.get_params(), b.get_params())
    a.close()
    b.close()
