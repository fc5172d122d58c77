"""The operator by itself as a chain of kernels: FP64 with two tiled wavelet
levels (layers of 128^2 and smaller ones of the least size and depth), with one
tiled level, and with every level on the layer's CTA (few CTAs), for each
number of filter taps; and several vectors at once.

Tolerances as in the parity tests: relative L2 error 1e-10 for FP64 and 1e-5
for FP32 against the FP64 oracle (the sums of the single-CTA transform in the
same order).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import Oracle  # noqa: E402
from synth import configs, random_vector  # noqa: E402

TOL = {"f64": 1e-10, "f32": 1e-5}


def rel(a, b):
    a, b = np.asarray(a, dtype=np.float64), np.asarray(b, dtype=np.float64)
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2011_06842_gb300 import build
    build.build()
    import paper_2011_06842_gb300 as P
    return P


def geometry(taps, layers):
    hs = np.linspace(0.0, 9000.0, len(layers))
    gs = [configs.GuideStar(1e-4, -5e-5, 90000.0), configs.GuideStar(-8e-5, 3e-5), configs.GuideStar(0.0, 1e-4)]
    return configs.Geometry("chain", D=17.0, obstruction=0.2, n_sub=37, gs=gs, wavelet_N=taps, r0=0.15,
                            layers=[configs.Layer(h, 1.0 / len(layers), n, J) for h, (n, J) in zip(hs, layers)],
                            wind=[(10.0, 0.3 * i) for i in range(len(layers))])


DEEP = [(128, 7), (32, 2), (64, 3)]      # two tiled levels in FP64
SHALLOW = [(128, 1), (64, 6), (32, 2)]   # one: a layer has a single level


@pytest.mark.parametrize("taps", [1, 2, 3, 4])
@pytest.mark.parametrize("layers,grid", [(DEEP, 0), (DEEP, 6), (DEEP, 5), (SHALLOW, 0)])
@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_operator(lib, taps, layers, grid, prec):
    geom = geometry(taps, layers)
    w = np.array([0.7, 1.3, 2.0])
    o, f = Oracle(geom, w), lib.Fewha(geom, w, prec, grid=grid)
    dt = f.dtype
    xs = np.stack([random_vector(o.n, seed) for seed in (1, 2, 3)])
    ref = np.stack([o.apply_op(x) for x in xs])
    xd = torch.tensor(xs, dtype=dt, device="cuda")
    assert rel(f.apply_op(xd[0]).cpu().numpy(), ref[0]) < TOL[prec]
    assert rel(f.apply_op_noalloc(xd[1]).cpu().numpy(), ref[1]) < TOL[prec]
    assert rel(f.apply_op_multi(xd).cpu().numpy(), ref) < TOL[prec]
    s = random_vector(f.n_slopes, 9)
    assert rel(f.rhs(torch.tensor(s, dtype=dt, device="cuda")).cpu().numpy(), o.rhs(s)) < TOL[prec]
    f.close()
