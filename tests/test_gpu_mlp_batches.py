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


def test_predictions_ask_for_activations_alone(binding):
    # 7-256-256-256-2 on 4 M rows: 777 BF16 activations a row, 6.2 GB; the gradients'
    # buffers (FP32 pre-activations, two layers' gradients) would be 18 GB more
    rows = 4_000_000
    x = torch.zeros((rows, 7), device="cuda")
    y = torch.empty((rows, 2), device="cuda")
    net = binding.MLP([7, 256, 256, 256, 2], seed=3)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    lib = binding.load_library()
    assert lib.mirage_mlp_forward(net.handle, x.data_ptr(), rows, y.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] <= rows * 777 * 2 + (64 << 20)
    net.close()


@pytest.mark.parametrize("dims", [[7, 48, 2], [5, 300, 33, 3], [7, 256, 256, 256, 2]])
def test_passes_of_changing_sizes(binding, dims):
    # predictions and gradients in turn, growing and shrinking: each as on a
    # network that does nothing else
    rng = np.random.default_rng(2)
    net = binding.MLP(dims, seed=4)
    for n, what in [(10, "f"), (200, "g"), (700, "f"), (150, "g"), (300, "g"), (900, "g"), (20, "f"), (1000, "f"), (900, "g")]:
        x = torch.as_tensor(rng.standard_normal((n, dims[0])).astype(np.float32), device="cuda")
        t = torch.as_tensor(rng.standard_normal((n, dims[-1])).astype(np.float32), device="cuda")
        other = binding.MLP(dims, seed=4)
        if what == "f":
            assert torch.equal(net.forward(x), other.forward(x)), n
        else:
            for a, b in zip(net.grad(x, t), other.grad(x, t)):
                assert torch.allclose(a, b, rtol=1e-12, atol=0), n  # (the loss is summed by atomics)
        other.close()
    net.train(x, t, 5, 64, 1e-3, seed=1)
    torch.cuda.synchronize()
    assert np.isfinite(net.get_params()).all()
    net.close()
