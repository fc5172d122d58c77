"""The P^T gather's two band plans in a batch: the library's choice (taller bands where a group has several per
CTA), heights set by the caller, and back.  Every launch equals the FP64 oracle (1e-10 in FP64, 1e-5 in FP32, as in
the parity tests: fixed-iteration time steps)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import Oracle  # noqa: E402
from synth import FrozenFlowSensors, configs  # noqa: E402


def rel(a, b):
    return np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b)


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2011_06842_gb300 import build
    build.build()
    import paper_2011_06842_gb300 as P
    return P


_sequences = {}


def sequence(name):
    """Geometry, slopes, weights and the oracle's solutions of two frames of four iterations."""
    if name not in _sequences:
        geom = configs.get(name)
        s, w = FrozenFlowSensors(geom, seed=41).sequence(2, seed=42)
        o = Oracle(geom, w)
        st, ref = o.new_state(4), []
        for t in range(2):
            o.solve(s[t].numpy(), st, max_iter=4, augmented=True)
            ref.append(st["c"].copy())
        _sequences[name] = (geom, s, w, ref)
    return _sequences[name]


@pytest.mark.parametrize("prec,tol", [("f64", 1e-10), ("f32", 1e-5)])
def test_heights_set_by_the_caller_hold_in_a_batch(lib, prec, tol):
    names, ctas = ["elt", "medium", "elt"], [9, 3, 40]
    handles = []
    for name in names:
        geom, s, w, ref = sequence(name)
        handles.append(lib.Fewha(geom, w, prec))

    def check(expected):
        batch = lib.FewhaBatch(handles, ctas)
        got = batch.pt_bands()
        states = [f.new_state(4) for f in handles]
        cs = [torch.zeros(f.n, dtype=f.dtype, device="cuda") for f in handles]
        for t in range(2):
            stats = batch.solve([sequence(n)[1][t].to(f.slope_dtype).cuda() for n, f in zip(names, handles)], cs,
                                states, max_iter=4)
            for name, c, r in zip(names, cs, batch.read_stats(stats)):
                assert r["status"] == 0 and rel(c.cpu().numpy(), sequence(name)[3][t]) < tol, (name, t)
        batch.close()
        assert got == expected, (got, expected)

    standard = [f.launch_info()["pt_bands"] for f in handles]  # 8 and 4 rows
    assert (handles[0].launch_info()["pt_rows_large"], handles[0].launch_info()["pt_rows_small"]) == (8, 4)
    batch = lib.FewhaBatch(handles, ctas)
    automatic = batch.pt_bands()
    batch.close()
    assert automatic[0] < standard[0] and automatic[1] < standard[1]  # several bands per CTA
    check(automatic)
    for f in handles:
        f.set_pt_bands(8, 4)
    check(standard)
    for f in handles:
        f.auto_pt_bands()
    check(automatic)
    for f in handles:
        f.close()


def test_autotuner_keeps_the_automatic_heights_apart(lib):
    """The heights the tuner names are those that run: None is the library's choice, (8, 4) the caller's."""
    geom, s, w, ref = sequence("medium")
    handles = [lib.Fewha(geom, w, "f32") for _ in range(2)]
    batch = lib.FewhaBatch(handles, [3, 3])
    automatic = batch.pt_bands()
    batch.close()
    standard = [f.launch_info()["pt_bands"] for f in handles]
    sd = s[0].float().cuda()

    def step(batch):
        batch.solve([sd, sd], [torch.zeros(f.n, device="cuda") for f in handles], [f.new_state(4) for f in handles],
                    max_iter=4)

    best, timings = lib.autotune_batch(handles, step, candidates=[([3, 3], None)], reps=1, tiles=(), bands=((8, 4),))
    assert len(timings) == 2  # the automatic heights and the caller's
    batch = lib.FewhaBatch(handles, [3, 3])
    assert batch.pt_bands() == (automatic if best["bands"][0] is None else standard)
    batch.close()
    for f in handles:
        f.close()


@pytest.mark.parametrize("name,prec,ctas,taller", [("ltao", "f32", 36, False), ("elt", "f64", 48, False),
                                                   ("elt", "f32", 40, False), ("elt", "f32", 9, True),
                                                   ("elt", "f32", 152, False), ("medium", "f32", 2, True),
                                                   ("medium", "f64", 20, True), ("tiny", "f64", 1, True)])
def test_taller_bands_where_they_pay(lib, name, prec, ctas, taller):
    """The library's choice on both sides of the line (each side was timed with both plans)."""
    geom = configs.get(name)
    f = lib.Fewha(geom, np.ones(len(geom.gs)), prec)
    batch = lib.FewhaBatch([f], [ctas])
    standard = f.launch_info()["pt_bands"]
    assert batch.pt_bands()[0] < standard if taller else batch.pt_bands()[0] == standard
    batch.close()
    f.close()
