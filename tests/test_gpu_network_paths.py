"""Paths of the warm-start network beside the ones of test_gpu_learned.py."""
import numpy as np
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


SPAN = 260 * 2.0 ** -24  # about as many FP32 additions one after another as a 16 x 16 tile has pixels, then FP64


def constant_gradients(value, B, H, W):
    """Weight gradient per tap and bias gradient of an input of ones and a constant output gradient."""
    rows, cols = [H - 1, H, H - 1], [W - 1, W, W - 1]
    return value * B * np.outer(rows, cols), value * B * H * W


@pytest.mark.parametrize("B,Cin,Cout,side", [(512, 5, 9, 64), (512, 32, 5, 64), (512, 4, 32, 64), (152, 6, 12, 32),
                                             (153, 6, 12, 32), (37, 40, 33, 72)])
def test_weight_gradient_of_many_images(B, Cin, Cout, side):
    """FP32 partial sums stay short however many images there are: an input of ones and a constant output
    gradient, whose sums have a closed form and whose rounding errors add up instead of cancelling.  Many tiles per
    partial, and on both sides of the line between one round of partials and several (1216 tiles of 16 x 8)."""
    from paper_2011_06842_gb300 import build, load_library
    build.build()
    L = load_library()
    hw = side * side
    x = torch.ones(B, Cin, side, side, device="cuda")
    g = torch.full((B, Cout, side, side), 0.1, device="cuda")
    size = L.fewha_conv3x3_wgrad_workspace(Cin, Cout, B, side, side)
    ws = torch.full((size + 64,), 7.0, device="cuda")
    gw, gb = torch.zeros(Cout, Cin, 3, 3, device="cuda"), torch.zeros(Cout, device="cuda")
    rw, rb = constant_gradients(float(g[0, 0, 0, 0]), B, side, side)
    for times, accumulate in ((1, 0), (2, 1)):
        assert L.fewha_conv3x3_bwd_weight(x.data_ptr(), Cin * hw, hw, Cin, g.data_ptr(), Cout * hw, hw, Cout, B, side,
                                          side, gw.data_ptr(), gb.data_ptr(), accumulate, ws.data_ptr(),
                                          torch.cuda.current_stream().cuda_stream) == 0
        assert np.abs(gw.cpu().numpy() / (times * rw) - 1).max() < SPAN
        assert np.abs(gb.cpu().numpy() / (times * rb) - 1).max() < SPAN
    assert torch.all(ws[size:] == 7.0)  # nothing written past the workspace


@pytest.mark.parametrize("offset", [0, 1])
def test_network_gradient_of_many_images(offset):
    """fewha_convnet_bwd with several rounds of partials in a workspace of the stated size, on either side of an
    8-byte boundary: hidden layers of ones, a last convolution that passes channel 0 on, and a constant output
    gradient have closed-form gradients of the second and third weights."""
    import ctypes as C

    from paper_2011_06842_gb300 import build, load_library
    from paper_2011_06842_gb300.fewha import NET
    build.build()
    L = load_library()
    groups = [(80, 64), (3, 32)]  # 2608 tiles
    n = sum(c * s * s for c, s in groups)
    dev = dict(device="cuda", dtype=torch.float32)
    w = [torch.zeros(32, 4, 3, 3, **dev), torch.zeros(32, 32, 3, 3, **dev), torch.zeros(5, 32, 3, 3, **dev)]
    w[2][0, :, 1, 1] = 1.0
    b = [torch.zeros(k, **dev) for k in (32, 32, 5)]
    gw, gb = [torch.zeros_like(t) for t in w], [torch.zeros_like(t) for t in b]
    hidden = [[f(c, 32, s, s, **dev) for c, s in groups] for f in (torch.ones, torch.ones, torch.empty, torch.empty)]
    N, off = NET(), 0
    N.C0, N.C, N.C3, N.ngroups = 4, 32, 5, len(groups)
    for i, (c, s) in enumerate(groups):
        N.count[i], N.side[i], N.off[i] = c, s, off
        off += c * s * s
        for dst, buf in zip((N.h1, N.h2, N.g1, N.g2), hidden):
            dst[i] = buf[i].data_ptr()
    for i in range(3):
        N.w[i], N.b[i], N.gw[i], N.gb[i] = (t[i].data_ptr() for t in (w, b, gw, gb))
    x, gy = torch.ones(4, n, **dev), torch.full((5, n), 0.1, **dev)
    size = min(152, sum(c * ((s + 15) // 16) ** 2 for c, s in groups)) * (32 * 32 * 9 + 32)
    ws = torch.full((size + 64,), 7.0, **dev)
    assert L.fewha_convnet_bwd(C.byref(N), x.data_ptr(), n, gy.data_ptr(), n, ws.data_ptr() + 4 * offset,
                               torch.cuda.current_stream().cuda_stream) == 0
    ref = [constant_gradients(float(gy[0, 0]), c, s, s) for c, s in groups]
    rw, rb = sum(r[0] for r in ref), sum(r[1] for r in ref)
    for got in (gw[1], gw[2]):
        assert np.abs(got.cpu().numpy() / rw - 1).max() < SPAN
    for got in (gb[1], gb[2]):
        assert np.abs(got.cpu().numpy() / rb - 1).max() < SPAN
    assert torch.all(ws[offset + size:] == 7.0) and torch.all(ws[:offset] == 7.0)


@pytest.mark.parametrize("runs", [8, 9, 16])
def test_many_runs_of_layer_sizes(runs):
    """As many runs of equal-size layers as one launch takes, and more (layer by layer then): forward and every
    parameter gradient against the FP64 oracle (FP32 1e-5 and 1e-4, as for two runs), and the tensor-core forward
    within bfloat16's reach of it (1e-2 of the norm, as for a single convolution).  The gradients after that
    forward belong to its own hidden layers: the oracle's gradients from those, again 1e-4."""
    from oracle import learned as OL
    layers = [configs.Layer(500.0 * i, 1.0 / runs, (16, 8)[i % 2], 2) for i in range(runs)]
    geom = configs.Geometry("runs", D=2.0, obstruction=0.0, n_sub=4, gs=[configs.GuideStar(0.0, 0.0)], layers=layers,
                            r0=0.2, wind=[(10.0, 0.1)] * runs)
    net = network(geom)
    assert len(net.groups) == runs
    rng = np.random.default_rng(12)
    x, gy = rng.standard_normal((4, net.n)), rng.standard_normal((5, net.n))
    xd, gd = (torch.tensor(a, dtype=torch.float32, device="cuda") for a in (x, gy))
    p, ref = net.params_numpy(), np.zeros((5, net.n))

    def gradients(hidden):
        total = {}
        for (off, cnt, nl), h in zip(net.groups, hidden):
            span = slice(off, off + nl * nl)
            parts = OL.net_backward(x[:, span].reshape(1, 4, nl, nl), p, h, gy[:, span].reshape(1, 5, nl, nl))
            for k, g in parts.items():
                total[k] = total.get(k, 0.0) + g
        return total

    hidden = []
    for off, cnt, nl in net.groups:
        out, h = OL.net_forward(x[:, off:off + nl * nl].reshape(1, 4, nl, nl), p)
        ref[:, off:off + nl * nl] = out.reshape(5, -1)
        hidden.append(h)
    exact = gradients(hidden)

    def rel(a, b):
        return np.linalg.norm(a - b) / np.linalg.norm(b)

    y = torch.full((5, net.n), 7.0, device="cuda")
    for tensor_cores, tol in ((False, 1e-5), (True, 1e-2), (False, 1e-5)):
        net.forward(xd.data_ptr(), net.n, y, tensor_cores=tensor_cores)
        assert rel(y.double().cpu().numpy(), ref) < tol
        net.backward(xd.data_ptr(), net.n, gd)
        got = net.grad.double().cpu().numpy()
        grads = exact
        if tensor_cores:
            grads = gradients([(a.double().cpu().numpy(), b.double().cpu().numpy()) for a, b in zip(net.h1, net.h2)])
        for name, (o, shape) in net.offsets.items():
            assert rel(got[o:o + int(np.prod(shape))].reshape(shape), grads[name]) < 1e-4, (name, tensor_cores)


@pytest.mark.parametrize("name", ["micro", "mixed", "elt"])
def test_one_launch_has_the_bits_of_three(name):
    """The whole network on the tensor cores in one launch adds the same products in the same order as its
    convolutions one by one."""
    net = network(configs.get(name))
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn(4, net.n, generator=g, device="cuda")
    y, z = torch.empty(5, net.n, device="cuda"), torch.empty(5, net.n, device="cuda")
    net.forward(x.data_ptr(), net.n, y, tensor_cores=True)
    for conv, _, launch in net.convolutions(x.data_ptr(), net.n, z, tensor_cores=True):
        assert launch() == 0, conv
    assert torch.equal(y, z)
