"""Operator calls in a CUDA graph: their kernels are joined by programmatic edges there.  Captured once and replayed
on new inputs, every result equals the uncaptured call's, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from synth import configs  # noqa: E402


@pytest.mark.parametrize("prec", ["f64", "f32", "bf16s"])
@pytest.mark.parametrize("name", ["elt", "tiny"])  # layers in the split and in the whole-layer form
def test_captured_operator_calls(name, prec):
    from paper_2011_06842_gb300 import Fewha, build
    from paper_2011_06842_gb300.fewha import McaoFit
    build.build()
    geom = configs.get(name)
    f = Fewha(geom, np.ones(len(geom.gs)), prec)
    mirrors = [(85, 0.5, 0.0), (47, 1.0, 4000.0)] if name == "elt" else [(21, 0.5, 0.0)]
    mc = McaoFit(f, mirrors, [(0.0, 0.0), (5e-5, 0.0)])
    g = torch.Generator(device="cuda").manual_seed(3)
    xs = torch.randn(4, 3, f.n, generator=g, device="cuda", dtype=f.dtype)
    ss = torch.randn(4, f.n_slopes, generator=g, device="cuda").to(f.slope_dtype)
    x, s = xs[0].clone(), ss[0].clone()
    y, b, a = torch.zeros(5, f.n, dtype=f.dtype, device="cuda"), torch.zeros_like(x[0]), f.new_mirror()
    m, start = mc.new_mirrors(), mc.new_mirrors()

    def calls():
        f.rhs(s, out=b)
        f.apply_op(x[0], out=y[0])
        f.apply_op_noalloc(x[1], out=y[1])
        f.apply_op_multi(x, out=y[2:])
        f.fit(x[0], out=a)
        m.copy_(start)
        mc.fit(x[1], m, 2)
        f.apply_op(y[0], out=x[2])  # a chain on the result of another

    calls()  # what is allocated on first use
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        calls()
    for i in range(4):
        results = []
        for run in (graph.replay, calls):
            x.copy_(xs[i])
            s.copy_(ss[i])
            for out in (y, b, a, m):
                out.fill_(7.0)
            run()
            results.append([t.clone() for t in (y, b, a, m, x[2])])
        for one, two in zip(*results):
            assert torch.equal(one, two), i
    mc.close()
    f.close()
