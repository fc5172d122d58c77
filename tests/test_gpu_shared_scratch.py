"""fewha_rhs beside fewha_fit and fewha_mcao_fit of the same handle on two
streams (the next frame's right-hand side while this frame is fitted): the
calls write no scratch buffer in common, so every result equals the one of the
same calls in order, bit for bit."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import numpy as np  # noqa: E402

from synth import configs  # noqa: E402


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_rhs_beside_the_fits(prec):
    from paper_2011_06842_gb300 import Fewha, build
    from paper_2011_06842_gb300.fewha import McaoFit
    build.build()
    geom = configs.elt()  # 128^2 and 64^2 layers: the split form's approximation scratch is in use on both sides
    f = Fewha(geom, np.ones(len(geom.gs)), prec)
    assert f.launch_info()["split_levels"] == 1
    mc = McaoFit(f, [(85, 0.5, 0.0), (47, 1.0, 4000.0)], [(0.0, 0.0), (5e-5, 0.0)])
    rounds = 40
    g = torch.Generator(device="cuda").manual_seed(3)
    s = torch.randn(rounds, f.n_slopes, generator=g, device="cuda", dtype=f.dtype)
    c = torch.randn(rounds, f.n, generator=g, device="cuda", dtype=f.dtype)
    out = {}
    for mode in ("in order", "beside"):
        b = torch.zeros(rounds, f.n, device="cuda", dtype=f.dtype)
        a = torch.zeros(rounds, f.fit(c[0]).numel(), device="cuda", dtype=f.dtype)
        m = torch.zeros(rounds, mc.n_actuators, device="cuda", dtype=f.dtype)
        torch.cuda.synchronize()
        s1 = torch.cuda.Stream()
        s2 = s1 if mode == "in order" else torch.cuda.Stream()
        for i in range(rounds):
            with torch.cuda.stream(s1):
                f.rhs(s[i], out=b[i])
            with torch.cuda.stream(s2):
                f.fit(c[i], out=a[i])
                mc.fit(c[i], m[i], 2)
        torch.cuda.synchronize()
        out[mode] = (b, a, m)
    for one, two in zip(out["in order"], out["beside"]):
        assert torch.equal(one, two)
    mc.close()
    f.close()
