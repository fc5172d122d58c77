"""Paths of the warm-start network beside the ones of test_gpu_learned.py."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from synth import configs  # noqa: E402


def network(geom, seed=3):
    from paper_2011_06842_gb300 import build
    build.build()
    from paper_2011_06842_gb300.learned import ConvNet
    return ConvNet(geom, seed=seed)


@pytest.mark.parametrize("tensor_cores", [False, True])
@pytest.mark.parametrize("name", ["medium", "elt"])
def test_output_over_the_input(name, tensor_cores):
    """y over the memory of x, as three launches per layer size allow: the outputs of a y of its own.  FP32: the
    same launches, bit for bit.  Tensor cores: the same bfloat16 operands and FP32 sums in one launch or three;
    a hidden value whose last bits differ may round to the neighbouring bfloat16, 2^-8 of one of 288 terms,
    hence 1e-4 of the output's norm."""
    net = network(configs.get(name))
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn(4, net.n, generator=g, device="cuda")
    y = torch.empty(5, net.n, device="cuda")
    net.forward(x.data_ptr(), net.n, y, tensor_cores=tensor_cores)
    both = torch.empty(5, net.n, device="cuda")
    both[:4].copy_(x)
    net.forward(both.data_ptr(), net.n, both, tensor_cores=tensor_cores)
    if tensor_cores:
        assert float((both - y).norm() / y.norm()) < 1e-4
    else:
        assert torch.equal(both, y)
    # newest first: the input's channels from the last row up
    both[1:].copy_(x.flip(0))
    net.forward(both[4].data_ptr(), -net.n, both, tensor_cores=tensor_cores)
    assert float((both - y).norm() / y.norm()) < 1e-4


def test_backward_after_replays_of_a_captured_forward():
    """A captured tensor-core forward replayed on new inputs, each followed by backward(): the gradients of the
    same calls without a graph (the same launches, bit for bit)."""
    net = network(configs.tiny())
    g = torch.Generator(device="cuda").manual_seed(1)
    xs = torch.randn(3, 4, net.n, generator=g, device="cuda")
    gy = torch.randn(5, net.n, generator=g, device="cuda")
    x, y = xs[0].clone(), torch.empty_like(gy)
    net.forward(x.data_ptr(), net.n, y, tensor_cores=True)  # everything the call needs is loaded before the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        net.forward(x.data_ptr(), net.n, y, tensor_cores=True)
    replayed = []
    for i in range(3):
        x.copy_(xs[i])
        graph.replay()
        net.backward(x.data_ptr(), net.n, gy)
        replayed.append(net.grad.clone())
    for i in range(3):
        x.copy_(xs[i])
        net.forward(x.data_ptr(), net.n, y, tensor_cores=True)
        net.backward(x.data_ptr(), net.n, gy)
        assert torch.equal(replayed[i], net.grad), i
