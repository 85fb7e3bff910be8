"""Device memory of the training calls of the warm-start network."""
import numpy as np
import pytest

from paper_1109_1146_gb300 import mf

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _net_and_data(c, shape, seed=3):
    N, H, W = shape
    rng = np.random.Generator(np.random.PCG64(seed))
    x, dy = (torch.from_numpy(rng.standard_normal((N, c, H, W)).astype(np.float32)).cuda() for _ in range(2))
    return mf.CNN(channels=c, seed=5), x, dy, torch.empty_like(x)


def test_a_forward_that_does_not_fit():
    # the buffers of the forward before are freed to make room: a backward has nothing to read, and the
    # network goes on with the next forward
    net, x, dy, y = _net_and_data(6, (1, 20, 24))
    net.forward(x, y)
    net.backward(x, dy)
    want_y, want_g = y.clone(), net.get_grads()
    side = 1 << 20  # 2^47 bytes per layer
    st = mf.load().mf_cnn_forward(net._h, x.data_ptr(), 1, side, side, y.data_ptr())
    assert st == mf.MF_ENOMEM
    with pytest.raises(mf.MFError) as e:
        net.backward(x, dy)
    assert e.value.status == mf.MF_EINVAL
    net.zero_grad()
    net.forward(x, y)
    net.backward(x, dy)
    assert torch.equal(y, want_y)
    np.testing.assert_array_equal(net.get_grads(), want_g)


@pytest.mark.parametrize("c", [6, 10])
def test_first_backward_allocates_nothing(c):
    # the first backward of a network can be captured in a CUDA graph, and adds the same gradients as a plain one
    shape = (2, 40, 33)
    ref, x, dy, y = _net_and_data(c, shape)
    ref.forward(x, y)
    ref.backward(x, dy)
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    net = mf.CNN(channels=c, seed=5, stream=side)
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        net.forward(x, y)
    side.synchronize()
    with torch.cuda.graph(graph, stream=side):
        net.backward(x, dy)
    graph.replay()
    torch.cuda.synchronize()
    np.testing.assert_array_equal(net.get_grads(), ref.get_grads())


def test_gradient_workspace_holds_what_the_largest_layer_writes():
    # one more training network takes its activations and the partial sums of 2 blocks per SM, 9248 floats each
    net, x, dy, y = _net_and_data(6, (1, 8, 8))
    net.forward(x, y)
    net.backward(x, dy)
    torch.cuda.synchronize()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    before = torch.cuda.mem_get_info()[0]
    other = mf.CNN(channels=6, seed=6)
    other.forward(x, y)
    other.backward(x, dy)
    torch.cuda.synchronize()
    # (allocations come in blocks of 2 MB: the workspace, parameters, activations, gradients)
    assert before - torch.cuda.mem_get_info()[0] <= 2 * sms * 9248 * 4 + 4 * (2 << 20)
