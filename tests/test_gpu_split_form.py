"""The solver's split form (the finest wavelet levels tiled over all CTAs) in every mode of a time step: recycling
of the last and of all directions, residual replacement, a right-hand side already in the state, residual-driven
stopping, the persistent kernel and the per-phase launches, batches, each filter length.  Small layers run the
whole-layer form, so the geometries here have one 128^2 layer beside smaller ones: in FP64 two tiled levels ("deep")
or one ("shallow", a layer with a single level), in FP32 one.

Bounds as in the parity tests: relative L2 error 1e-10 (FP64) and 1e-5 (FP32) of the solution after each time step,
ten times that of the residual, or 100 times the oracle's own sensitivity to slopes perturbed by the precision's
rounding unit where that is more; FP32 with the residual replaced divides by ||r|| / ||b|| (r = b - M c is formed in
FP32, so its rounding is relative to ||b||)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import Oracle  # noqa: E402
from synth import FrozenFlowSensors, configs  # noqa: E402

TOL = {"f64": 1e-10, "f32": 1e-5}
UNIT = {"f64": 2.0 ** -53, "f32": 2.0 ** -24}
LAYERS = {"deep": [(128, 5), (32, 2), (64, 3)], "shallow": [(128, 1), (64, 4), (32, 2)]}
FRAMES = 3

MODES = {
    "last": dict(),
    "plain": dict(augmented=False),
    "all": dict(recycle_all=True),
    "replace": dict(true_res_every=2),
    "all, replace": dict(recycle_all=True, true_res_every=2),
    "stop": dict(rtol=2e-2, max_iter=60),
    "stop, replace": dict(rtol=2e-2, max_iter=60, true_res_every=3),
}


def rel(a, b):
    a, b = np.asarray(a, dtype=np.float64), np.asarray(b, dtype=np.float64)
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2011_06842_gb300 import build
    build.build()
    import paper_2011_06842_gb300 as P
    return P


def geometry(name, taps=3):
    layers = LAYERS[name]
    gs = [configs.GuideStar(1e-4, -5e-5, 90000.0), configs.GuideStar(-8e-5, 3e-5), configs.GuideStar(0.0, 1e-4)]
    return configs.Geometry("split_" + name, D=17.0, obstruction=0.2, n_sub=37, gs=gs, wavelet_N=taps, r0=0.15,
                            layers=[configs.Layer(h, 1.0 / 3, n, J) for h, (n, J) in zip((0.0, 4500.0, 9000.0), layers)],
                            wind=[(10.0, 0.3 * i) for i in range(3)])


_problems, _references = {}, {}


def problem(name, taps=3):
    if (name, taps) not in _problems:
        geom = geometry(name, taps)
        s, w = FrozenFlowSensors(geom, seed=23).sequence(FRAMES, seed=24)
        _problems[name, taps] = (geom, s.numpy(), w, Oracle(geom, w))
    return _problems[name, taps]


def reference(name, taps, mode, prec):
    """Per frame: the oracle's solution, residual, iterations, ||r|| / ||b|| and the two bounds."""
    key = (name, taps, mode, prec)
    if key not in _references:
        geom, s, w, o = problem(name, taps)
        m = dict(MODES[mode])
        kw = dict(loop_mode=Oracle.LOOP_ALL if m.pop("recycle_all", False) else Oracle.LOOP_LAST, **m)
        its, rtol = kw.pop("max_iter", 5), kw.pop("rtol", 0.0)
        rng = np.random.default_rng(6)
        a, b, out = o.new_state(8), o.new_state(8), []
        for t in range(FRAMES):
            r = o.solve(s[t], a, max_iter=its, rtol=rtol, **kw)
            o.solve(s[t] * (1 + UNIT[prec] * rng.standard_normal(s[t].shape)), b, max_iter=r["iterations"], **kw)
            tol = TOL[prec] / r["rel_res"] if prec == "f32" and kw.get("true_res_every") else TOL[prec]
            out.append((a["c"].copy(), a["r_prev"].copy(), r["iterations"], r["rel_res"],
                        max(tol, 100 * rel(b["c"], a["c"])), max(10 * tol, 100 * rel(b["r_prev"], a["r_prev"]))))
        _references[key] = out
    return _references[key]


def check(stats, c, state, ref):
    cr, rr, its, _, tc, tr = ref
    assert stats["status"] == 0 and stats["iterations"] == its
    assert rel(c.cpu().numpy(), cr) < tc
    assert rel(state.r_prev.cpu().numpy(), rr) < tr


def split_handle(lib, name, prec, taps=3, grid=0):
    geom, s, w, o = problem(name, taps)
    f = lib.Fewha(geom, w, prec, grid=grid)
    assert f.launch_info()["split_levels"] == 1
    return f, torch.tensor(s, dtype=f.slope_dtype, device="cuda")


@pytest.mark.parametrize("persistent", [True, False])
@pytest.mark.parametrize("mode", sorted(MODES))
@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("name", sorted(LAYERS))
def test_time_steps(lib, name, prec, mode, persistent):
    f, s = split_handle(lib, name, prec)
    st, c = f.new_state(8), torch.zeros(f.n, dtype=f.dtype, device="cuda")
    kw = dict(max_iter=5)
    kw.update(MODES[mode])
    for t, ref in enumerate(reference(name, 3, mode, prec)):
        check(f.read_stats(f.solve(s[t], c, st, persistent=persistent, **kw)), c, st, ref)
    f.close()


@pytest.mark.parametrize("grid", [6, 7])
@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("name", sorted(LAYERS))
def test_fewest_ctas(lib, name, prec, grid):
    """Twice as many CTAs as layers, and one more."""
    f, s = split_handle(lib, name, prec, grid=grid)
    st, c = f.new_state(8), torch.zeros(f.n, dtype=f.dtype, device="cuda")
    for t, ref in enumerate(reference(name, 3, "all, replace", prec)):
        check(f.read_stats(f.solve(s[t], c, st, 5, recycle_all=True, true_res_every=2)), c, st, ref)
    f.close()


@pytest.mark.parametrize("taps", [1, 2, 4])
@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("name", sorted(LAYERS))
def test_filter_lengths(lib, name, prec, taps):
    f, s = split_handle(lib, name, prec, taps)
    for persistent in (True, False):
        st, c = f.new_state(8), torch.zeros(f.n, dtype=f.dtype, device="cuda")
        for t, ref in enumerate(reference(name, taps, "replace", prec)):
            check(f.read_stats(f.solve(s[t], c, st, 5, persistent=persistent, true_res_every=2)), c, st, ref)
    f.close()


@pytest.mark.parametrize("mode", ["last", "replace"])
@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("name", sorted(LAYERS))
def test_right_hand_side_in_the_state(lib, name, prec, mode):
    """b and the warm-restart residual folded into the state by the caller, as a deflated warm start leaves it."""
    f, s = split_handle(lib, name, prec)
    for persistent in (True, False):
        st, c = f.new_state(8), torch.zeros(f.n, dtype=f.dtype, device="cuda")
        for t, ref in enumerate(reference(name, 3, mode, prec)):
            b = f.rhs(s[t])
            st.r_prev.copy_((b - st.b_prev) + st.r_prev)
            st.b_prev.copy_(b)
            check(f.read_stats(f.solve(None, c, st, 5, rhs_in_state=True, persistent=persistent, **MODES[mode])), c, st,
                  ref)
    f.close()


@pytest.mark.parametrize("mode", ["last", "all", "all, replace", "stop", "stop, replace"])
@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_batch(lib, prec, mode):
    """Split groups (six CTAs or more for three layers), a whole-layer group of the same geometry and groups of
    several sizes in one launch."""
    names, ctas = ["deep", "shallow", "deep", "deep", "shallow"], [6, 11, 40, 5, 1]
    handles = [lib.Fewha(problem(n)[0], problem(n)[2], prec) for n in names]
    slopes = [torch.tensor(problem(n)[1], dtype=handles[0].slope_dtype, device="cuda") for n in names]
    batch = lib.FewhaBatch(handles, ctas)
    assert batch.ctas() == ctas
    states = [f.new_state(8) for f in handles]
    cs = [torch.zeros(f.n, dtype=f.dtype, device="cuda") for f in handles]
    kw = dict(max_iter=5)
    kw.update(MODES[mode])
    for t in range(FRAMES):
        stats = batch.read_stats(batch.solve([s[t] for s in slopes], cs, states, **kw))
        for n, c, st, r in zip(names, cs, states, stats):
            check(r, c, st, reference(n, 3, mode, prec)[t])
    batch.close()
    for f in handles:
        f.close()
