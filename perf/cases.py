"""The work that users of the library have it do, as measurable cases.

Every case is a dict of plain values: the kind of call, the telescope (pupil,
sensors, guide stars, layers), the precision and the options.  The listed
cases are the configurations of this repository (an 8 m, a 16 m and a 39 m
telescope, LTAO and MCAO asterisms, a batch of 64 instances, the network of
the learned warm start); ``draw`` gives further telescopes in between, with
odd sensor sizes, guide-star and layer counts among them.

Kinds of calls
  step      one time step of the reconstructor loop: ``Fewha.solve`` on the next
            frame of a frozen-flow sequence, warm-started from the last one
  loop      a whole closed-loop step of Algorithm 3: pseudo-open-loop slopes,
            solve, fitting, gain control
  batch     one time step of many instances in one captured launch
  apply     y = M x (condition numbers, users' own solvers)
  multi     y_v = M x_v for several vectors (deflation directions)
  rhs       b = W^{-T} A^T C^{-1} s
  mcao      fitting onto three deformable mirrors, warm-started
  predict   the network's inference on the last four solutions
  train     one training step of the network (forward, backward, Adam)

``exact`` restates each of them in FP64 with dense one-dimensional
interpolation and wavelet matrices, without the library.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch
import torch.nn.functional as F

ARCSEC = math.pi / 648000.0
FRAMES = 4          # frames that a prepared sequence cycles through
FRAME_RATE = 500.0  # [Hz]
TYPES = {"f64": torch.float64, "f32": torch.float32, "bf16s": torch.float32}
SLOPE_TYPES = {"f64": torch.float64, "f32": torch.float32, "bf16s": torch.bfloat16}
CHANNELS = (4, 32, 32, 5)  # the learned warm start's network
MIRRORS = ((85, 0.5, 0.0), (47, 1.0, 4000.0), (53, 1.0, 12700.0))  # actuators per side, pitch [m], altitude [m]

# Telescopes of this repository's configurations: pupil, central obstruction,
# sensor size, laser and natural guide stars on rings (radius in arcsec; sizes
# of low-order natural-star sensors as n_low x 2x2 and 1x1), layers from the
# ground to `top` metres on `grid`^2 nodes up to 8 km and `grid_high`^2 above.
TINY = dict(D=8.0, obstruction=0.0, n_sub=16, lgs=0, lgs_radius=0.0, ngs=4, ngs_radius=30.0, low_order=False,
            layers=2, top=8000.0, grid=32, grid_high=32, J=3, r0=0.15)
MEDIUM = dict(D=16.0, obstruction=0.2, n_sub=40, lgs=4, lgs_radius=45.0, ngs=0, ngs_radius=0.0, low_order=False,
              layers=5, top=12000.0, grid=64, grid_high=64, J=4, r0=0.15)
ELT = dict(D=39.0, obstruction=0.28, n_sub=84, lgs=6, lgs_radius=60.0, ngs=0, ngs_radius=0.0, low_order=False,
           layers=9, top=16000.0, grid=128, grid_high=64, J=5, r0=0.129)
LTAO = dict(ELT, n_sub=80, lgs_radius=225.0, ngs=3, ngs_radius=300.0)
MCAO = dict(ELT, lgs_radius=80.0, ngs=3, ngs_radius=60.0, low_order=True)


def listed():
    return [
        # smallest call: an 8 m telescope's time step, plain PCG at full precision
        dict(TINY, name="step_8m_f64", kind="step", precision="f64", augmented=False, k=4, iterations=4),
        # an ordinary one: a 16 m telescope, augmented PCG
        dict(MEDIUM, name="step_16m_f32", kind="step", precision="f32", augmented=True, k=8, iterations=6),
        # the headline: an ELT time step, augmented PCG (the counts are fixed, as in the paper's real-time loop)
        dict(ELT, name="step_elt_f32", kind="step", precision="f32", augmented=True, k=8, iterations=6),
        # the same operator at full precision, the paper's iteration count
        dict(ELT, name="step_elt_f64", kind="step", precision="f64", augmented=True, k=8, iterations=4),
        # a whole closed-loop step of the LTAO asterism (wide field, natural and laser stars, 80x80 sensors)
        dict(LTAO, name="loop_ltao_f32", kind="loop", precision="f32", augmented=True, k=8, iterations=4),
        # many telescopes of uneven size in one launch
        dict(name="batch_64_f32", kind="batch", precision="f32", augmented=True, k=8, iterations=6, tiny=24, medium=24,
             elt=16),
        # the operator by itself, as the condition-number diagnostics apply it
        dict(ELT, name="apply_elt_f64", kind="apply", precision="f64"),
        # the operator on the five directions of a deflated warm start
        dict(ELT, name="multi_elt_f32", kind="multi", precision="f32", vectors=5),
        # right-hand side with 16-bit slopes, sensors of different sizes (MCAO)
        dict(MCAO, name="rhs_mcao_bf16s", kind="rhs", precision="bf16s"),
        # MCAO fitting onto the paper's three mirrors, 4 CG iterations
        dict(ELT, name="mcao_fit_f32", kind="mcao", precision="f32", directions=7, iterations=4),
        # inference and training of the warm-start network on ELT layers
        dict(ELT, name="predict_elt", kind="predict", precision="f32"),
        dict(ELT, name="train_elt", kind="train", precision="f32"),
    ]


def _draw_telescope(rng, largest=84):
    """A telescope between the 8 m and the 39 m one: subapertures of 0.4-0.5 m."""
    n_sub = int(round(math.exp(rng.uniform(math.log(12), math.log(largest)))))
    D = round(n_sub * rng.uniform(0.4, 0.5), 2)
    grid = 32 if n_sub <= 20 else 64 if n_sub <= 42 else 128
    lgs, ngs = rng.choice([(0, 3), (0, 5), (3, 0), (4, 0), (5, 1), (6, 0), (6, 3)])
    # the coarsest block keeps at least 4 x 4 coefficients on the largest layers: the sensors do not see a lone mean
    deepest = {32: 3, 64: 4, 128: 5}[grid]
    return dict(D=D, obstruction=rng.choice([0.0, 0.2, 0.28]), n_sub=n_sub, lgs=lgs,
                lgs_radius=float(rng.randint(50, 110)) if lgs else 0.0, ngs=ngs,
                ngs_radius=float(rng.randint(20, 60)) if ngs else 0.0, low_order=False,
                layers=rng.randint(2, 9), top=float(rng.randint(8, 16)) * 1000.0, grid=grid,
                grid_high=64 if grid == 128 else grid, J=rng.randint(deepest - 1, deepest), r0=0.14)


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "loop", "batch", "apply", "multi", "rhs", "mcao", "predict",
                       "train"])
    if kind == "batch":
        return dict(kind=kind, precision="f32", augmented=True, k=rng.choice([4, 8]), iterations=rng.randint(3, 6),
                    tiny=rng.randint(1, 24), medium=rng.randint(1, 24), elt=rng.randint(0, 12))
    if kind == "mcao":
        return dict(ELT, kind=kind, precision=rng.choice(["f32", "f32", "f64"]), directions=rng.randint(3, 9),
                    iterations=rng.randint(1, 6), n_sub=rng.randint(60, 84))
    case = dict(_draw_telescope(rng), kind=kind)
    if kind in ("predict", "train"):
        case["precision"] = "f32"
    elif kind == "rhs":
        case["precision"] = rng.choice(["f64", "f32", "bf16s"])
        case["low_order"] = case["ngs"] == 3
    else:
        case["precision"] = rng.choice(["f64", "f32", "f32"])
    if kind in ("step", "loop"):
        case["augmented"] = rng.random() < 0.7
        case["k"] = rng.choice([3, 4, 8])
        case["iterations"] = rng.randint(2, 10 if case["precision"] == "f64" else 6)
    if kind == "multi":
        case["vectors"] = rng.randint(1, 8)
    return case


# --- telescopes and inputs ----------------------------------------------------
def _geometry(case):
    """Guide stars, layers and winds from the case's numbers."""
    gs = []
    for count, radius, H in ((case["ngs"], case["ngs_radius"], 0.0), (case["lgs"], case["lgs_radius"], 90000.0)):
        for i in range(count):
            a = 2 * math.pi * i / count + (0.3 if H == 0.0 and case["lgs"] else 0.0)
            low = (2, 1, 1)[i % 3] if case["low_order"] and H == 0.0 else 0
            gs.append(SimpleNamespace(theta_x=radius * ARCSEC * math.cos(a), theta_y=radius * ARCSEC * math.sin(a), H=H,
                                      n_sub=low))
    L = case["layers"]
    hs = [case["top"] * i / (L - 1) for i in range(L)]
    w = [math.exp(-h / 4000.0) for h in hs]
    layers = [SimpleNamespace(h=h, cn2=wi / sum(w), n=case["grid"] if h <= 8000.0 else case["grid_high"], J=case["J"],
                              delta=1.0) for h, wi in zip(hs, w)]
    rng = np.random.default_rng(1000 + L)
    wind = list(zip(rng.uniform(5.0, 20.0, L), rng.uniform(0.0, 2 * math.pi, L)))
    return SimpleNamespace(D=case["D"], obstruction=case["obstruction"], n_sub=case["n_sub"], gs=gs, layers=layers,
                           r0=case["r0"], L0=25.0, alpha=2.0, wavelet_N=3, wind=wind,
                           n=sum(l.n * l.n for l in layers), sizes=[g.n_sub or case["n_sub"] for g in gs])


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _rng(seed):
    g = torch.Generator(device=_device())
    g.manual_seed(int(seed))
    return g


def _randn(g, *shape, dtype=torch.float64):
    return torch.randn(*shape, generator=g, device=_device(), dtype=dtype)


def _lit(geom, ns):
    if ns == 1:
        return torch.ones(1, 1, dtype=torch.bool, device=_device())
    x = -geom.D / 2 + (torch.arange(ns, dtype=torch.float64, device=_device()) + 0.5) * geom.D / ns
    r = torch.sqrt(x[:, None] ** 2 + x[None, :] ** 2)
    return (r >= geom.obstruction * geom.D / 2) & (r <= geom.D / 2)


def _sensor_frames(geom, seed, frames=FRAMES, snr=10.0):
    """Shack-Hartmann slopes of a frozen-flow von Karman sky: (frames, n_slopes)
    in FP64 and the noise weights 1/sigma_g^2.  A subaperture measures the
    difference of the mean phase on its opposite edges, plus white noise."""
    dev, f64 = _device(), torch.float64
    g = _rng(seed)
    step = geom.D / geom.n_sub / 2
    reach = max(geom.D / 2 + max(abs(s.theta_x), abs(s.theta_y)) * l.h for s in geom.gs for l in geom.layers)
    M = 64
    while M < 2 * reach / step + 8:
        M *= 2
    f = torch.fft.fftfreq(M, step, dtype=f64, device=dev)
    psd = 0.023 * (f[:, None] ** 2 + f[None, :] ** 2 + 1.0 / geom.L0 ** 2) ** (-11.0 / 6.0)
    psd[0, 0] = 0.0
    screens = []
    for lay in geom.layers:
        amp = torch.sqrt(psd * (geom.r0 * lay.cn2 ** -0.6) ** (-5.0 / 3.0)) / (M * step)
        screens.append(torch.fft.ifft2(torch.complex(_randn(g, M, M), _randn(g, M, M)) * amp).real * M * M)
    t = torch.arange(frames, dtype=f64, device=dev).reshape(-1, 1, 1, 1) / FRAME_RATE
    third = torch.tensor([1.0, 3.0, 5.0], dtype=f64, device=dev) / 6.0

    def phase(star, x, y):
        total = torch.zeros((frames,) + x.shape, dtype=f64, device=dev)
        for lay, screen, (speed, direction) in zip(geom.layers, screens, geom.wind):
            cone = 1.0 - lay.h / star.H if star.H > 0 else 1.0
            u = (cone * x + star.theta_x * lay.h - speed * math.cos(direction) * t) / step
            v = (cone * y + star.theta_y * lay.h - speed * math.sin(direction) * t) / step
            iu, iv = torch.floor(u), torch.floor(v)
            fu, fv = u - iu, v - iv
            iu, iv = iu.long() % M, iv.long() % M
            ju, jv = (iu + 1) % M, (iv + 1) % M
            total += (1 - fv) * ((1 - fu) * screen[iv, iu] + fu * screen[iv, ju]) + fv * (
                (1 - fu) * screen[jv, iu] + fu * screen[jv, ju])
        return total

    slopes, weights = [], []
    for star, ns in zip(geom.gs, geom.sizes):
        ds = geom.D / ns
        node = -geom.D / 2 + torch.arange(ns + 1, dtype=f64, device=dev) * ds
        edge = node[:-1, None] + third * ds
        V = phase(star, node[None, :, None].expand(ns, ns + 1, 3), edge[:, None, :].expand(ns, ns + 1, 3)).mean(-1)
        H = phase(star, edge[None, :, :].expand(ns + 1, ns, 3), node[:, None, None].expand(ns + 1, ns, 3)).mean(-1)
        s = torch.cat([(V[:, :, 1:] - V[:, :, :-1]).reshape(frames, -1), (H[:, 1:] - H[:, :-1]).reshape(frames, -1)], 1)
        lit = _lit(geom, ns).reshape(-1).repeat(2)
        sigma = s[0][lit].square().mean().sqrt().item() / snr
        slopes.append(s + sigma * _randn(g, *s.shape))
        weights.append(1.0 / sigma ** 2)
    return torch.cat(slopes, 1), np.array(weights)


def _prior(geom):
    """alpha * D, and the class (layer, band) of every coefficient with two
    sampled coefficients per axis and class."""
    ad, samples = [], []
    for l, lay in enumerate(geom.layers):
        n, J = lay.n, lay.J
        d = _spacing(geom, lay)
        kappa = 2.0 ** (-(11.0 / 3.0) * J) / (0.5 * 6.88 * (d / (geom.r0 * lay.cn2 ** -0.6)) ** (5.0 / 3.0))
        level = np.zeros((n, n))
        bands = [(0, 0, n >> J)]
        for s in range(1, J + 1):
            nb = (n >> J) << (s - 1)
            for r, q in ((0, nb), (nb, 0), (nb, nb)):
                level[r:r + nb, q:q + nb] = s
                bands.append((r, q, nb))
        ad.append((geom.alpha * kappa * 2.0 ** ((11.0 / 3.0) * level)).reshape(-1))
        for r, q, nb in bands:
            offs = sorted({nb // 4, 3 * nb // 4})
            samples.append((l, r, q, nb, [(r + a, q + b) for a in offs for b in offs]))
    return torch.tensor(np.concatenate(ad), device=_device()), samples


def _solutions(geom, seed, frames):
    """Layer coefficients with the prior's spectrum, slowly changing from frame to frame (FP64)."""
    ad, _ = _prior(geom)
    g = _rng(seed)
    c, out = _randn(g, geom.n), []
    for _ in range(frames):
        out.append(c / torch.sqrt(ad))
        c = 0.98 * c + 0.2 * _randn(g, geom.n)
    return torch.stack(out)


def _mirror_shapes(geom, seed, frames):
    """Smooth ground-mirror shapes (a few low orders), (frames, (n_sub+1)^2)."""
    x = torch.linspace(-1, 1, geom.n_sub + 1, dtype=torch.float64, device=_device())
    g = _rng(seed)
    polys = torch.stack([x ** i for i in range(4)])
    return torch.stack([torch.einsum("ij,ia,jb->ab", _randn(g, 4, 4), polys, polys).reshape(-1) for _ in range(frames)])


def _ground_slopes(geom, a):
    """Gamma a for every sensor (all of the geometry's size): the mirror's own slopes."""
    m = geom.n_sub + 1
    sx, sy = _gamma(a.reshape(-1, m, m))
    one = torch.cat([sx.flatten(1), sy.flatten(1)], 1)
    return one.repeat(1, len(geom.gs))


def _batch_parts(case):
    """Instances of the batch: (telescope, how many, CTAs each, round)."""
    parts = []
    if case["elt"]:
        parts.append((ELT, case["elt"], max(1, min(9, 144 // case["elt"])), 0))
    rest = 1 if case["elt"] else 0
    parts.append((MEDIUM, case["medium"], max(1, min(6, (144 - case["tiny"]) // case["medium"])), rest))
    parts.append((TINY, case["tiny"], 1, rest))
    return parts


def _batch_frames(case, seed):
    """Per instance (telescope, CTAs, round, slopes (FRAMES, n), weights); instances of one telescope share its weights."""
    out = []
    for p, (tel, count, ctas, rnd) in enumerate(_batch_parts(case)):
        geom = _geometry(tel)
        for i in range(count):
            s, w = _sensor_frames(geom, 1000 * seed + 100 * p + i, frames=2)
            if i == 0:
                first = w
            out.append((geom, ctas, rnd, s, first))
    return out


def _directions(count):
    """Fitting directions: the axis and a ring of 0.25 arcmin."""
    return [(0.0, 0.0)] + [(15 * ARCSEC * math.cos(2 * math.pi * i / (count - 1)),
                            15 * ARCSEC * math.sin(2 * math.pi * i / (count - 1))) for i in range(count - 1)]


# --- prepare and run ------------------------------------------------------------
def prepare(case, seed):
    from paper_2011_06842_gb300 import Fewha, FewhaBatch
    from paper_2011_06842_gb300.fewha import McaoFit
    from paper_2011_06842_gb300.learned import ConvNet, LearnedWarmStart
    kind, prec = case["kind"], case["precision"]
    st = SimpleNamespace(case=case, i=0)
    dtype = TYPES[prec]
    if kind == "batch":
        parts = _batch_frames(case, seed)
        st.f = [Fewha(g, w, prec) for g, _, _, _, w in parts]
        st.batch = FewhaBatch(st.f, [p[1] for p in parts], [p[2] for p in parts])
        st.frames = [torch.cat([p[3][t].to(dtype) for p in parts]) for t in range(2)]
        st.slopes = torch.zeros_like(st.frames[0])
        sizes = [f.n for f in st.f]
        # vectors start on 16-byte boundaries: every n is a multiple of 4
        st.c = torch.zeros(sum(sizes), dtype=dtype, device=_device())
        st.states = [f.new_state(case["k"]) for f in st.f]
        st.stats = st.batch.bind(list(st.slopes.split([f.n_slopes for f in st.f])), list(st.c.split(sizes)), st.states,
                                 case["iterations"], augmented=case["augmented"])
        st.graph = st.batch.capture_graph()
        return st
    geom = _geometry(case)
    if kind == "predict":
        st.net = ConvNet(geom, seed=seed % 1000)
        x = _solutions(geom, seed, 8)
        ad, _ = _prior(geom)
        st.ring = (x * torch.sqrt(ad)).float().contiguous()
        st.y = torch.zeros((CHANNELS[-1], geom.n), dtype=torch.float32, device=_device())
        return st
    s, w = _sensor_frames(geom, seed)
    st.f = f = Fewha(geom, w, prec)
    if kind in ("step", "loop"):
        st.frames = s
        if kind == "loop":
            st.a = _mirror_shapes(geom, seed + 1, FRAMES + 1).to(dtype).contiguous()
            st.frames = s - _ground_slopes(geom, st.a[:FRAMES].double())
            st.pol = torch.zeros(f.n_slopes, dtype=SLOPE_TYPES[prec], device=_device())
            st.fit, st.next = f.new_mirror(), f.new_mirror()
        st.frames = st.frames.to(SLOPE_TYPES[prec]).contiguous()
        st.c = torch.zeros(f.n, dtype=dtype, device=_device())
        st.state = f.new_state(case["k"])
        st.stats = f.new_stats()
    elif kind in ("apply", "multi"):
        st.x = [_solutions(geom, seed + t, case.get("vectors", 1)).to(dtype).contiguous() for t in range(2)]
        st.y = torch.zeros_like(st.x[0])
    elif kind == "rhs":
        st.frames = s.to(SLOPE_TYPES[prec]).contiguous()
        st.b = torch.zeros(f.n, dtype=dtype, device=_device())
    elif kind == "mcao":
        st.c = _solutions(geom, seed, FRAMES).to(dtype).contiguous()
        st.fit = McaoFit(f, MIRRORS, _directions(case["directions"]))
        st.a = st.fit.new_mirrors()
    elif kind == "train":
        st.c = _solutions(geom, seed, 5 + FRAMES).float().contiguous()
        st.learned = LearnedWarmStart(f, geom, seed=seed % 1000)
    return st


def run(st):
    case, i = st.case, st.i
    kind = case["kind"]
    st.i = i + 1
    if kind == "batch":
        st.slopes.copy_(st.frames[i % 2])
        st.graph.replay()
        return {"c": st.c}
    if kind == "predict":
        j = i % 4
        st.net.forward(st.ring[j + 4].data_ptr(), -st.ring.shape[1], st.y, tensor_cores=True)
        return {"y": st.y}
    f = st.f
    if kind == "step":
        f.solve(st.frames[i % FRAMES], st.c, st.state, case["iterations"], augmented=case["augmented"], stats=st.stats)
        return {"c": st.c, "r": st.state.r_prev, "b": st.state.b_prev, "P": st.state.P, "Q": st.state.Q}
    if kind == "loop":
        t = i % FRAMES
        f.pol_slopes(st.frames[t], st.a[t], out=st.pol)
        f.solve(st.pol, st.c, st.state, case["iterations"], augmented=case["augmented"], stats=st.stats)
        f.fit(st.c, out=st.fit)
        f.control(True, 0.4, st.a[t], st.a[t + 1], st.fit, out=st.next)
        return {"c": st.c, "r": st.state.r_prev, "b": st.state.b_prev, "fit": st.fit, "next": st.next}
    if kind == "apply":
        return {"y": f.apply_op(st.x[i % 2][0], out=st.y[0])}
    if kind == "multi":
        return {"y": f.apply_op_multi(st.x[i % 2], out=st.y)}
    if kind == "rhs":
        return {"b": f.rhs(st.frames[i % FRAMES], out=st.b)}
    if kind == "mcao":
        return {"a": st.fit.fit(st.c[i % FRAMES], st.a, case["iterations"])}
    net = st.learned.net
    st.learned.train_step(st.c, 3 + i % FRAMES, 1e-3)
    return {"y": st.learned.y, "grad": net.grad, "param": net.param}


# --- the least work of one pass ---------------------------------------------------
def _telescope_work(geom, case, iterations):
    """Bytes of a time step's inputs, outputs and state, and the operator's
    floating-point operations (stencils and short filters) over all iterations."""
    w = 8 if case["precision"] == "f64" else 4
    sw = 2 if case["precision"] == "bf16s" else w
    n, slopes = geom.n, sum(2 * ns * ns for ns in geom.sizes)
    nodes, L = sum((ns + 1) ** 2 for ns in geom.sizes), len(geom.layers)
    basis = min(case.get("k", 0), iterations)
    # slopes, c, r, b and the two diagonals; the recycled directions read (augmented) and written
    vectors = 2 + 2 * 3 + 2 * basis * (2 if case.get("augmented") else 1)
    transform = 2 * 2 * 6 * n * 4 // 3  # two passes of 6-tap filters, levels 1 + 1/4 + ...
    project = nodes * L * 9             # one bilinear sample per node and layer
    op = 2 * transform + 2 * project + 4 * slopes + 2 * nodes
    flops = iterations * (op + 14 * n) + transform + project + slopes
    return vectors * n * w + slopes * sw, flops, op


def work(case):
    kind = case["kind"]
    if kind == "batch":
        total = [0, 0]
        for tel, count, _, _ in _batch_parts(case):
            b, fl, _ = _telescope_work(_geometry(tel), case, case["iterations"])
            total[0] += count * b
            total[1] += count * fl
        return {"bytes": total[0], "flops": total[1]}
    geom = _geometry(case)
    w = 8 if case["precision"] == "f64" else 4
    n = geom.n
    if kind in ("predict", "train"):
        macs = n * 9 * sum(a * b for a, b in zip(CHANNELS, CHANNELS[1:]))
        params = sum(9 * a * b + b for a, b in zip(CHANNELS, CHANNELS[1:]))
        if kind == "predict":
            return {"bytes": 4 * (n * (CHANNELS[0] + CHANNELS[-1]) + params), "flops": 2 * macs}
        # forward, data gradient (not of the first layer) and weight gradient
        first = n * 9 * CHANNELS[0] * CHANNELS[1]
        return {"bytes": 4 * (5 * n + 2 * n + 8 * params), "flops": 2 * (3 * macs - first)}
    b, fl, op = _telescope_work(geom, case, case.get("iterations", 1))
    if kind in ("step", "loop"):
        return {"bytes": b, "flops": fl}
    if kind in ("apply", "multi"):
        v = case.get("vectors", 1)
        return {"bytes": (2 * v + 1) * n * w, "flops": v * op}
    if kind == "rhs":
        sw = 2 if case["precision"] == "bf16s" else w
        return {"bytes": n * w + sum(2 * ns * ns for ns in geom.sizes) * sw, "flops": op // 2}
    acts = sum(d[0] ** 2 for d in MIRRORS)
    nodes = case["directions"] * (geom.n_sub + 1) ** 2
    return {"bytes": (n + 2 * acts) * w,
            "flops": 2 * 2 * 6 * n * 4 // 3 + nodes * 9 * (len(geom.layers) + len(MIRRORS))
            + case["iterations"] * (2 * 9 * len(MIRRORS) * nodes + 10 * acts)}


# --- the same in FP64, from dense one-dimensional matrices ------------------------
def _taps():
    """Daubechies-3 low-pass filter (spectral factorisation, roots inside the unit circle)."""
    poly = np.array([1.0])
    for y in np.roots([6.0, 3.0, 1.0]):  # P_3(y) = 1 + 3 y + 6 y^2
        a = 1.0 - 2.0 * y
        d = np.sqrt(a * a - 1.0 + 0j)
        z = a + d if abs(a + d) < 1 else a - d
        poly = np.convolve(poly, [1.0, -z])
    for _ in range(3):
        poly = np.convolve(poly, [1.0, 1.0])
    h = np.real(poly)
    return h * math.sqrt(2.0) / h.sum()


def _spacing(geom, lay):
    R = max((1.0 - lay.h / s.H if s.H > 0 else 1.0) * geom.D / 2 + max(abs(s.theta_x * lay.h), abs(s.theta_y * lay.h))
            for s in geom.gs)
    return R / (lay.n / 2 - 2)


def _hat(coords, n):
    """Dense linear-interpolation matrix (len(coords), n) for positions in grid units."""
    k = torch.floor(coords)
    f = coords - k
    A = torch.zeros((len(coords), n), dtype=torch.float64, device=_device())
    rows = torch.arange(len(coords), device=_device())
    A[rows, k.long()] = 1.0 - f
    A[rows, k.long() + 1] = f
    return A


def _gamma(phi):
    """Gradient of pupil-node phases (..., m, m): x and y slopes (..., m-1, m-1)."""
    a, b, c, d = phi[..., :-1, :-1], phi[..., :-1, 1:], phi[..., 1:, :-1], phi[..., 1:, 1:]
    return 0.5 * ((b - a) + (d - c)), 0.5 * ((c - a) + (d - b))


class _Operator:
    """M, its parts and the preconditioner of one telescope in FP64; vectors are (batch, n)."""

    def __init__(self, geom, weights):
        self.geom, self.dev = geom, _device()
        h = _taps()
        g = [(-1) ** t * h[5 - t] for t in range(6)]
        self.W = {}
        N = 2
        while N <= max(l.n for l in geom.layers):
            A = np.zeros((N, N))
            for k in range(N // 2):
                for t in range(6):
                    A[k, (2 * k + t) % N] += h[t]
                    A[N // 2 + k, (2 * k + t) % N] += g[t]
            self.W[N] = torch.tensor(A, device=self.dev)
            N *= 2
        self.proj = []
        for s, ns in zip(geom.gs, geom.sizes):
            x = -geom.D / 2 + torch.arange(ns + 1, dtype=torch.float64, device=self.dev) * (geom.D / ns)
            self.proj.append([])
            for lay in geom.layers:
                cone = 1.0 - lay.h / s.H if s.H > 0 else 1.0
                d = _spacing(geom, lay)
                self.proj[-1].append(tuple(_hat((cone * x + th * lay.h) / d + lay.n / 2, lay.n)
                                           for th in (s.theta_y, s.theta_x)))
        self.weight = [_lit(geom, ns).double() * w for ns, w in zip(geom.sizes, weights)]
        self.ad, self.samples = _prior(geom)

    def layers(self, c):
        return [v.reshape(-1, l.n, l.n) for v, l in
                zip(c.split([l.n * l.n for l in self.geom.layers], dim=1), self.geom.layers)]

    def inverse(self, x, J):
        x = x.clone()
        n = x.shape[-1]
        for t in range(J - 1, -1, -1):
            N = n >> t
            x[:, :N, :N] = self.W[N].T @ x[:, :N, :N] @ self.W[N]
        return x

    def forward(self, x, J):
        x = x.clone()
        n = x.shape[-1]
        for t in range(J):
            N = n >> t
            x[:, :N, :N] = self.W[N] @ x[:, :N, :N] @ self.W[N].T
        return x

    def adjoint(self, slopes):
        """W^{-T} A^T C^{-1} s; slopes: per guide star (x, y) of shape (batch, ns, ns)."""
        out = [0.0] * len(self.geom.layers)
        for g, (sx, sy) in enumerate(slopes):
            vx, vy = 0.5 * self.weight[g] * sx, 0.5 * self.weight[g] * sy
            psi = torch.zeros(vx.shape[0], vx.shape[1] + 1, vx.shape[2] + 1, dtype=vx.dtype, device=vx.device)
            psi[:, :-1, :-1] += -vx - vy
            psi[:, :-1, 1:] += vx - vy
            psi[:, 1:, :-1] += -vx + vy
            psi[:, 1:, 1:] += vx + vy
            for l, (Ay, Ax) in enumerate(self.proj[g]):
                out[l] = out[l] + Ay.T @ psi @ Ax
        return torch.cat([self.forward(u, lay.J).flatten(1) for u, lay in zip(out, self.geom.layers)], 1)

    def slopes(self, nodal, only=None):
        """Gamma P of nodal layers (`only`: the one layer that is not zero)."""
        out = []
        for g in range(len(self.geom.gs)):
            phi = 0.0
            for l, (Ay, Ax) in enumerate(self.proj[g]):
                if only is None:
                    phi = phi + Ay @ nodal[l] @ Ax.T
                elif l == only:
                    phi = Ay @ nodal @ Ax.T
            out.append(_gamma(phi))
        return out

    def nodal(self, c):
        return [self.inverse(x, lay.J) for x, lay in zip(self.layers(c), self.geom.layers)]

    def apply(self, c):
        return self.adjoint(self.slopes(self.nodal(c))) + self.ad * c

    def rhs(self, s):
        parts = []
        for v, ns in zip(s.split([2 * ns * ns for ns in self.geom.sizes], dim=1), self.geom.sizes):
            parts.append((v[:, :ns * ns].reshape(-1, ns, ns), v[:, ns * ns:].reshape(-1, ns, ns)))
        return self.adjoint(parts)

    def inv_jacobi(self):
        """Diagonal of alpha D + the mean of the data term's diagonal over sampled coefficients of each band."""
        J = [d.clone() for d in self.layers(self.ad[None])]
        todo = {}
        for l, r, q, nb, at in self.samples:
            todo.setdefault(l, []).append((r, q, nb, at))
        for l, bands in todo.items():
            lay = self.geom.layers[l]
            places = [p for _, _, _, at in bands for p in at]
            e = torch.zeros(len(places), lay.n, lay.n, dtype=torch.float64, device=self.dev)
            for i, (r, q) in enumerate(places):
                e[i, r, q] = 1.0
            diag = 0.0
            for (sx, sy), w in zip(self.slopes(self.inverse(e, lay.J), only=l), self.weight):
                diag = diag + (w * (sx * sx + sy * sy)).sum((1, 2))
            i = 0
            for r, q, nb, at in bands:
                J[l][0, r:r + nb, q:q + nb] += diag[i:i + len(at)].mean()
                i += len(at)
        return 1.0 / torch.cat([j.reshape(-1) for j in J])

    def first_step(self, s, iterations, inv_jacobi):
        """PCG from a zero state (batch of slopes): c, r, b and the directions p, q."""
        b = self.rhs(s)
        c, r = torch.zeros_like(b), b.clone()
        z = inv_jacobi * r
        p, rz = z.clone(), (r * z).sum(1, keepdim=True)
        ps, qs = [], []
        for _ in range(iterations):
            q = self.apply(p)
            ps.append(p)
            qs.append(q)
            alpha = rz / (p * q).sum(1, keepdim=True)
            c = c + alpha * p
            r = r - alpha * q
            z = inv_jacobi * r
            new = (r * z).sum(1, keepdim=True)
            p, rz = z + (new / rz) * p, new
        return c, r, b, ps, qs


def _exact_basis(case, vectors):
    """The bank that a first time step fills: iteration i in slot i mod k."""
    bank = torch.zeros(2, case["k"], vectors[0].shape[1], dtype=torch.float64, device=vectors[0].device)
    for i, v in enumerate(vectors):
        bank[1, i % case["k"]] = v[0]
    return bank


def _exact_mcao(case, geom, op, c):
    """CG on the normal equations of the fit, from zero mirrors."""
    x = -geom.D / 2 + torch.arange(geom.n_sub + 1, dtype=torch.float64, device=_device()) * (geom.D / geom.n_sub)
    dirs = _directions(case["directions"])
    hats = [[tuple(_hat((x + th * h) / pitch + (n - 1) / 2, n) for th in (ty, tx)) for n, pitch, h in MIRRORS]
            for tx, ty in dirs]
    y = []
    nodal = op.nodal(c[None])
    for tx, ty in dirs:
        phi = 0.0
        for lay, v in zip(geom.layers, nodal):
            d = _spacing(geom, lay)
            Ay, Ax = (_hat((x + th * lay.h) / d + lay.n / 2, lay.n) for th in (ty, tx))
            phi = phi + Ay @ v[0] @ Ax.T
        y.append(phi)

    def project(a):
        parts = [v.reshape(d[0], d[0]) for v, d in zip(a.split([d[0] ** 2 for d in MIRRORS]), MIRRORS)]
        return [sum(Ay @ v @ Ax.T for (Ay, Ax), v in zip(h, parts)) for h in hats]

    def adjoint(maps):
        return torch.cat([sum(h[k][0].T @ m @ h[k][1] for h, m in zip(hats, maps)).reshape(-1)
                          for k in range(len(MIRRORS))])

    r = adjoint(y)
    a, p, rr = torch.zeros_like(r), r.clone(), r @ r
    for _ in range(case["iterations"]):
        q = adjoint(project(p))
        alpha = rr / (p @ q)
        a, r = a + alpha * p, r - alpha * q
        new = r @ r
        p, rr = r + (new / rr) * p, new
    return a


def _net_weights(geom, seed):
    """The network's initial parameters (He initialisation from the seed, small last layer), in order w1 b1 w2 b2 w3 b3."""
    rng = np.random.default_rng(seed)
    out = []
    for i, (a, b) in enumerate(zip(CHANNELS, CHANNELS[1:])):
        gain = 0.1 if i == 2 else 1.0
        w = (rng.standard_normal(b * a * 9) * gain * math.sqrt(2.0 / (a * 9))).astype(np.float32)
        out += [torch.tensor(w.reshape(b, a, 3, 3), device=_device()).double().requires_grad_(),
                torch.zeros(b, dtype=torch.float64, device=_device(), requires_grad=True)]
    return out


def _net(geom, params, x):
    """y (5, n) from x (4, n): the layers of one grid size are a batch."""
    outs = []
    for lay, v in zip(geom.layers, x.split([l.n * l.n for l in geom.layers], dim=1)):
        h = v.reshape(1, -1, lay.n, lay.n)
        for i in range(3):
            h = F.conv2d(h, params[2 * i], params[2 * i + 1], padding=1)
            if i < 2:
                h = torch.relu(h)
        outs.append(h.reshape(CHANNELS[-1], -1))
    return torch.cat(outs, 1)


def exact(case, seed):
    kind = case["kind"]
    prec = case["precision"]
    if kind == "batch":
        done, out = {}, []
        for geom, _, _, s, w in _batch_frames(case, seed):
            key = (geom.D, tuple(w))
            if key not in done:
                op = _Operator(geom, w)
                done[key] = (op, op.inv_jacobi())
            op, ij = done[key]
            out.append(op.first_step(s[:1].float().double(), case["iterations"], ij)[0][0])
        return {"c": torch.cat(out)}
    geom = _geometry(case)
    if kind in ("predict", "train"):
        params = _net_weights(geom, seed % 1000)
        ad, _ = _prior(geom)
        if kind == "predict":
            x = (_solutions(geom, seed, 8) * torch.sqrt(ad)).float().double()
            with torch.no_grad():
                return {"y": _net(geom, params, x[[4, 3, 2, 1]])}
        c = _solutions(geom, seed, 5 + FRAMES).float().double()
        white = torch.sqrt(ad)
        y = _net(geom, params, c[[3, 2, 1, 0]] * white)
        t0 = (c[4] - c[3]) * white
        group = []
        for lay in geom.layers:
            m = torch.arange(lay.n, device=_device())
            m = torch.maximum(m[:, None], m[None, :])
            group.append((1 + (m >= lay.n // 8).int() + (m >= lay.n // 4).int() + (m >= lay.n // 2).int()).reshape(-1))
        group = torch.cat(group)
        target = torch.stack([t0] + [torch.where(group == k, t0, torch.zeros_like(t0)) for k in (1, 2, 3, 4)])
        ((y - target) ** 2).mean().backward()
        grad = torch.cat([p.grad.reshape(-1) for p in params])
        flat = torch.cat([p.detach().reshape(-1) for p in params])
        # Adam's first step: m / (1 - beta1) = g, v / (1 - beta2) = g^2
        return {"y": y.detach(), "grad": grad, "param": flat - 1e-3 * grad / (grad.abs() + 1e-8)}
    s, w = _sensor_frames(geom, seed)
    op = _Operator(geom, w)
    if kind in ("step", "loop"):
        frames = s
        if kind == "loop":
            a = _mirror_shapes(geom, seed + 1, FRAMES + 1).to(TYPES[prec]).double()
            frames = s - _ground_slopes(geom, a[:FRAMES])
        first = frames[:1].to(SLOPE_TYPES[prec]).double()
        if kind == "loop":
            first = first + _ground_slopes(geom, a[:1])
        c, r, b, ps, qs = op.first_step(first, case["iterations"], op.inv_jacobi())
        out = {"c": c[0], "r": r[0], "b": b[0]}
        if kind == "step":
            return dict(out, P=_exact_basis(case, ps), Q=_exact_basis(case, qs))
        x = -geom.D / 2 + torch.arange(geom.n_sub + 1, dtype=torch.float64, device=_device()) * (geom.D / geom.n_sub)
        fit = 0.0
        for lay, v in zip(geom.layers, op.nodal(c)):
            A = _hat(x / _spacing(geom, lay) + lay.n / 2, lay.n)
            fit = fit + A @ v[0] @ A.T
        fit = fit.reshape(-1)
        return dict(out, fit=fit, next=a[1] + 0.4 * (fit - a[0]))
    if kind in ("apply", "multi"):
        x = _solutions(geom, seed, case.get("vectors", 1)).to(TYPES[prec]).double()
        y = op.apply(x)
        return {"y": y[0] if kind == "apply" else y}
    if kind == "rhs":
        return {"b": op.rhs(s[:1].to(SLOPE_TYPES[prec]).double())[0]}
    return {"a": _exact_mcao(case, geom, op, _solutions(geom, seed, FRAMES)[0].to(TYPES[prec]).double())}
