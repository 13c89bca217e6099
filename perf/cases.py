"""Timed work of the library, through its public Python entry points.

Three kinds of case:

* ``forward``: a medium that a program has built once is set back to a saved
  state (``Medium.load_state``), advanced by ``steps`` time steps
  (``Medium.run``) and read back (receiver traces and the pressure field): one
  shot of a simulation campaign, or one leg of a checkpointed run;
* ``gradient``: the same start, then ``Medium.gradient`` (forward run,
  recomputation and discrete adjoint) for dL/dc and dL/dalpha0;
* ``serve``: a batch of requests through ``Server`` until all are done.

The media are those of the repository's workloads: 3 MHz, 12 points per
wavelength, CFL 0.4, Voronoi tissue maps with 2 % jitter (or a homogeneous or
two-layer map), an absorbing layer, a source line or aperture below it and
receivers two planes further down.  The saved state is a superposition of
plane waves over the whole grid, as in the middle of a run, not the zero field.

``exact`` repeats the same discrete scheme in plain float64 torch.
"""
import math

import numpy as np
import torch

import paper_2606_11103_gb300 as fw

F0 = 3e6
C0, RHO0 = 1540.0, 1000.0
AMP = 1e3                        # Pa

# Relaxation sets calibrated at 1-20 MHz (2, 3 and 4 mechanisms):
# alpha0, y, kappa1, kappa2, d1, alpha1, d2, alpha2
SETS = {
    2: [
        (0.5, 1.1, 0.98915, 0.99919, (1.5655e6, 46795.), (2.6493e8, 2.0205e7), (1.5839e5, 17082.), (6.233e7, 4.6994e6)),
        (1.09, 1.0, 0.98251, 0.99809, (2.5785e5, 2.0618e6), (5.9323e7, 2.4427e8), (37413., 89419.),
         (4.323e6, 1.9148e7)),
        (0.6, 1.5, 0.98, 0.98, (1.1105e7, 2608.8), (3.0306e8, 3.144e8), (2.9321e5, 37937.), (4.9282e7, 1.0098e7)),
        (0.25, 1.2, 0.99349, 0.99872, (1.0102e5, 8363.4), (6.5433e7, 5.0848e6), (1.3131e6, 27080.),
         (2.8883e8, 2.1299e7)),
    ],
    3: [
        (0.5, 1.1, 0.98016, 0.99992, (86220., 3.1317e5, 7.7826e7), (4.2535e7, 1.1781e8, 1.3839e10),
         (32523., 4.1149e6, 13572.), (1.556e7, 5.9028e8, 3.9279e6)),
        (1.09, 1.0, 0.99299, 0.98326, (3.5413e6, 4.5107e5, 59524.), (4.4229e8, 1.0667e8, 1.4179e7),
         (4.6522e6, 1.471e5, 28852.), (1.8651e9, 3.9078e7, 3.4755e6)),
        (0.6, 1.5, 0.98, 0.98, (34200., 2.927e5, 15579.), (3.7298e9, 4.9255e7, 3.6894e8),
         (2.2101e6, 8.8796e6, 36771.), (3.1423e8, 3.0461e8, 1.0092e7)),
        (0.25, 1.2, 0.98123, 0.98011, (32378., 4.9072e8, 24375.), (1.1588e8, 1.5305e10, 2.0484e7),
         (83992., 9.0544e5, 7925.2), (6.0823e7, 2.6463e8, 4.9482e6)),
        (0.75, 1.3, 0.98222, 0.98363, (1.3002e5, 4.8595e5, 43364.), (3.655e7, 9.1605e7, 1.4374e7),
         (8.4525e6, 1.0255e5, 15010.), (3.8511e8, 1.5678e11, 4.0093e6)),
        (0.15, 1.0, 0.99715, 0.99993, (19127., 54021., 3663.4), (3.8321e7, 9.897e7, 3.3426e6),
         (4.3951e5, 8085.6, 697.36), (3.8075e8, 1.4575e7, 6.4374e6)),
    ],
    4: [
        (0.5, 1.1, 0.98828, 0.99844, (1018.2, 2.502e5, 78287., 30110.), (8.7336e10, 1.038e8, 3.9756e7, 1.4989e7),
         (2.6333e6, 1.3768e5, 1.532e6, 13254.), (4.4727e8, 2.886e8, 3.354e10, 3.8553e6)),
        (1.09, 1.0, 0.99102, 0.98149, (40186., 5.3408e8, 28235., 2.9583e9), (8.8724e8, 6.4487e11, 3.3968e6, 4.9175e11),
         (1.2469e5, 3.4436e5, 2.7712e6, 53638.), (3.5505e7, 9.0398e7, 3.3735e8, 1.3488e7)),
        (0.6, 1.5, 0.98012, 0.98468, (1.0365e7, 2.7261e5, 7.9985e6, 3.2567e5), (2.9727e8, 4.8437e7, 9.2471e9, 3.303e8),
         (38252., 8.7927e5, 11429., 37265.), (2.7712e9, 1.1419e9, 9.6009e9, 9.9295e6)),
        (0.25, 1.2, 0.98485, 0.98084, (32538., 18238., 56251., 4.6078e7), (2.4704e11, 1.6747e7, 4.6167e7, 2.7812e9),
         (2.6326e5, 6.3487e7, 3.7677e7, 6508.7), (1.3478e8, 8.4142e9, 6.988e9, 4.3122e6)),
        (0.75, 1.3, 0.98003, 0.98084, (1.1002e7, 91593., 2877.6, 3.5878e5), (1.0229e10, 2.3747e7, 1.4647e5, 6.8948e7),
         (2.4972e6, 52229., 1.179e7, 24029.), (2.4705e8, 1.5579e8, 7.0855e8, 6.7401e6)),
        (0.15, 1.0, 0.98727, 0.98004, (110., 21795., 2.0325e5, 15183.), (5.3985e6, 3.0112e10, 2.4832e8, 3.2112e7),
         (6572.6, 38046., 1.3429e9, 3467.1), (1.2598e7, 7.8777e7, 4.4214e10, 3.2068e6)),
        (0.4, 0.8, 0.99338, 0.9903, (17217., 15192., 88168., 4.7756e5), (1.3412e7, 9.3504e8, 1.0237e8, 7.8051e9),
         (34121., 1.492e9, 5.1371e5, 11640.), (3.7136e7, 1.2876e11, 4.3852e8, 3.0512e6)),
        (0.9, 1.4, 0.98, 0.98, (261.96, 1.0439e7, 74149., 4.0334e5), (4.1721e8, 2.9001e8, 1.6957e7, 5.5736e7),
         (29472., 2.5098e5, 731.45, 16874.), (9.5714e11, 2.9808e8, 3.3067e8, 4.1653e6)),
    ],
}


# ---------------------------------------------------------------------------
# cases


def _case(name, kind, nz, ny, nx, mech, steps, medium="voronoi", storage="f32", order=2, pml=20, transition=0,
          nonlinear=False, ppw=12, cfl=0.4, checkpoint=0, requests=0):
    c = dict(kind=kind, nz=nz, ny=ny, nx=nx, mech=mech, steps=steps, medium=medium, storage=storage, order=order,
             pml=pml, transition=transition, nonlinear=nonlinear, ppw=ppw, cfl=cfl, checkpoint=checkpoint,
             requests=requests)
    return dict(c, name=name) if name else c


def listed():
    """nz = 0: a 2D grid [ny][nx]."""
    return [
        # the smallest workload: a homogeneous 256^2 plane, where each launch counts
        _case("plane_256", "forward", 0, 256, 256, 2, 256, medium="homogeneous"),
        # the calibration's plane-wave run: D = 10, W = 50 wavelengths at 16 points, two-stage layers of 3 wavelengths
        _case("protocol_360x992", "forward", 0, 360, 992, 2, 192, medium="homogeneous", pml=48, transition=48, ppw=16,
              cfl=0.2),
        # two-layer nonlinear plane with the thicker layer
        _case("two_layer_2048", "forward", 0, 2048, 2048, 4, 64, medium="two_layer", pml=30, nonlinear=True),
        # the smallest volume of the request stream
        _case("volume_128", "forward", 128, 128, 128, 4, 128),
        # a ragged volume with a transition layer, three mechanisms
        _case("ragged_231x187x301", "forward", 231, 187, 301, 3, 64, pml=12, transition=6),
        # the benchmark's volume
        _case("volume_512", "forward", 512, 512, 512, 4, 64),
        # 16-bit memory variables: binary16 on the largest side of the request stream, bfloat16 on an odd volume
        _case("volume_384_f16", "forward", 384, 384, 384, 4, 64, storage="f16"),
        _case("ragged_250x203x333_bf16", "forward", 250, 203, 333, 4, 64, storage="bf16"),
        # the fourth-order-in-time stencil
        _case("time_space_256", "forward", 256, 256, 256, 4, 64, order=4),
        # gradients: the inversion workload's plane (checkpoints every 32 steps) and a volume
        _case("gradient_1024", "gradient", 0, 1024, 1024, 3, 128, checkpoint=32),
        _case("gradient_volume_128", "gradient", 128, 128, 128, 2, 48, checkpoint=16),
        # continuous batching: planes of 512^2 and volumes of 128^3 in one queue
        _case("serve_8", "serve", 128, 512, 512, 4, 96, requests=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Sides 192 .. 2048 in 2D and 96 .. 384 in 3D, mostly odd, two to four
    mechanisms, every storage, both time schemes, with and without transition
    layer and nonlinearity; gradients on grids up to 1200^2 and 150^3."""
    kind = rng.choice(["forward", "forward", "forward", "forward", "gradient", "gradient", "serve"])
    if kind == "serve":
        return _case(None, "serve", rng.choice([96, 128, 160]), *[_log_int(rng, 384, 900)] * 2, rng.choice([2, 3, 4]),
                     rng.randint(64, 160), requests=rng.randint(4, 10))
    d3 = rng.random() < 0.6
    mech = rng.choice([2, 3, 4])
    pml = rng.randint(8, 24)
    transition = rng.choice([0, 0, rng.randint(4, 12)])
    if kind == "gradient":
        shape = [_log_int(rng, 80, 150) for _ in range(3)] if d3 else [0] + [_log_int(rng, 256, 1200) for _ in range(2)]
        return _case(None, kind, *shape, mech, rng.randint(24, 64) if d3 else rng.randint(48, 128), pml=pml,
                     transition=transition, checkpoint=rng.choice([0, 16, 25]))
    storage = rng.choice(["f32", "f32", "f32", "bf16", "f16", "f64"])
    top = (384 if d3 else 2048) if storage != "f64" else (160 if d3 else 640)
    shape = [_log_int(rng, 96, top) for _ in range(3)] if d3 else [0] + [_log_int(rng, 192, top) for _ in range(2)]
    return _case(None, kind, *shape, mech, rng.randint(48, 160), storage=storage, order=rng.choice([2, 2, 4]), pml=pml,
                 transition=transition, nonlinear=rng.random() < 0.3)


# ---------------------------------------------------------------------------
# inputs


def _shape(case):
    return (case["nz"], case["ny"], case["nx"]) if case["nz"] else (case["ny"], case["nx"])


def _grid(case):
    """(dx, dt)"""
    c_ref, c_top = (1450.0, 1580.0) if case["medium"] == "two_layer" else \
        (C0, C0) if case["medium"] == "homogeneous" else (C0, 1600.0 * 1.06)
    dx = c_ref / (F0 * case["ppw"])
    return dx, case["cfl"] * dx / c_top


def _maps(case, shape, seed, dev):
    """Sound speed, density, class index, beta (or None) and the rows of SETS the classes are."""
    rng = np.random.default_rng([seed, 1])
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    rows = SETS[case["mech"]]
    if case["medium"] == "homogeneous":
        one = torch.ones(shape, device=dev)
        return C0 * one, RHO0 * one, torch.zeros(shape, dtype=torch.int16, device=dev), None, [rows[rng.integers(len(rows))]]
    if case["medium"] == "two_layer":
        low = (torch.arange(shape[0], device=dev) >= shape[0] // 2).reshape([-1] + [1] * (len(shape) - 1)).expand(shape)
        pick = lambda a, b: torch.where(low, torch.tensor(b, device=dev), torch.tensor(a, device=dev)).contiguous()
        return (pick(1580.0, 1450.0), pick(1060.0, 950.0), low.to(torch.int16).contiguous(),
                pick(3.5, 6.0) if case["nonlinear"] else None, rows[1:3])
    # Voronoi tissue map: nearest of 64 (3D) or 32 (2D) seeds
    n_seed = 64 if len(shape) == 3 else 32
    seeds = rng.uniform(0.0, 1.0, (n_seed, len(shape))) * np.asarray(shape)
    owner = rng.integers(0, len(rows), n_seed)
    axes = [(torch.arange(n, device=dev) + 0.5).reshape([-1 if a == b else 1 for b in range(len(shape))])
            for a, n in enumerate(shape)]
    best = torch.full(shape, math.inf, device=dev)
    cls = torch.zeros(shape, dtype=torch.int16, device=dev)
    for s, o in zip(seeds, owner):
        near = sum((x - float(v)) ** 2 for x, v in zip(axes, s))
        closer = near < best
        best = torch.where(closer, near, best)
        cls.masked_fill_(closer, int(o))
    del best, near, closer
    c = torch.from_numpy(rng.uniform(1450.0, 1600.0, len(rows)).astype(np.float32)).to(dev)[cls.int()]
    rho = torch.from_numpy(rng.uniform(900.0, 1100.0, len(rows)).astype(np.float32)).to(dev)[cls.int()]
    for m in (c, rho):
        m *= 1.0 + 0.02 * torch.randn(shape, generator=gen, device=dev).clamp_(-3.0, 3.0)
    beta = torch.full(shape, 3.5, device=dev) + 0.5 * cls if case["nonlinear"] else None
    return c, rho, cls, beta, rows


def _waves(case, shape, seed, dev):
    """Initial pressure and velocities: eight plane waves of 10 to 24 cells per wavelength over the whole grid."""
    rng = np.random.default_rng([seed, 2])
    f = [torch.zeros(shape, device=dev) for _ in range(1 + len(shape))]
    for _ in range(8):
        n = rng.standard_normal(len(shape))
        n /= np.linalg.norm(n)
        k = 2.0 * math.pi / rng.uniform(10.0, 24.0)
        a, ph = AMP * rng.uniform(0.2, 0.5), rng.uniform(0.0, 2.0 * math.pi)
        arg = sum((float(k * v) * torch.arange(m, device=dev)).reshape([-1 if i == j else 1 for j in range(len(shape))])
                  for i, (m, v) in enumerate(zip(shape, n)))
        w = torch.cos(arg + ph)
        f[0].add_(w, alpha=a)
        for d in range(len(shape)):         # v_0 is along x, the last array axis
            f[1 + d].add_(w, alpha=a * float(n[len(shape) - 1 - d]) / (RHO0 * C0))
    return f


def _source(case, shape, seed, dx, dt):
    """Source mask, waveforms, waveform of each source, receiver mask."""
    rng = np.random.default_rng([seed, 3])
    w, nd = case["pml"] + case["transition"], len(shape)
    row = w + 4
    src, rcv = np.zeros(shape, np.uint8), np.zeros(shape, np.uint8)
    if nd == 2:                             # a line, 64 receivers on a row below it
        src[row] = 1
        rcv[row + 8, np.linspace(w + 4, shape[1] - w - 5, 64).round().astype(int)] = 1
    else:                                   # an aperture of half the lateral extent, receivers on every eighth cell
        lat = [slice(n // 4, n // 4 + n // 2) for n in shape[1:]]
        src[(row, *lat)] = 1
        rcv[(row + 2, *[slice(s.start, s.stop, 8) for s in lat])] = 1
    n_wave = 1 if nd == 2 else 8
    t = np.arange(case["steps"]) * dt
    delay = rng.uniform(0.0, 1.0 / F0, n_wave)[:, None] + 1.0 / F0
    rate = 2.0 * AMP * dx ** (nd - 1) / (RHO0 * C0)
    waves = rate * np.sin(2 * math.pi * F0 * (t - delay)) * np.exp(-((t - delay) * F0) ** 2)
    n_src = int(src.sum())
    return src, waves.astype(np.float32), (np.arange(n_src) * n_wave // n_src).astype(np.int32), rcv


def _parts(case):
    """The single simulations of a serve case: planes and volumes in turn."""
    return [dict(case, kind="forward", nz=case["nz"] if k % 2 else 0, ny=case["nz"] if k % 2 else case["ny"],
                 nx=case["nz"] if k % 2 else case["nx"]) for k in range(case["requests"])]


def _medium(case, seed, dev):
    shape = _shape(case)
    dx, dt = _grid(case)
    c, rho, cls, beta, rows = _maps(case, shape, seed, dev)
    classes = [fw.relax_params(*r[2:]) for r in rows]
    m = fw.Medium.from_classes(shape, dx, c, rho, cls, classes, dt=dt, beta=beta, pml=case["pml"],
                               transition=case["transition"], f0=F0, storage=case["storage"], time_order=case["order"])
    src, waves, wave_of, rcv = _source(case, shape, seed, dx, dt)
    m.set_sources(src, waves, wave_of)
    m.set_receivers(rcv, case["steps"])
    for k, f in enumerate(_waves(case, shape, seed, dev)):
        m.write_field(fw.FW_FIELD_P if k == 0 else fw.FW_FIELD_V, max(k - 1, 0), f)
    start = torch.empty(m.state_bytes(), dtype=torch.uint8, device=dev)
    m.save_state(out=start)
    alpha0 = torch.tensor([r[0] for r in rows], device=dev)[cls.int()] if case["kind"] == "gradient" else None
    return m, start, alpha0, int(rcv.sum())


def _weights(case, n_rcv, seed, dev):
    """dL/dtraces of a gradient."""
    gen = torch.Generator(device=dev).manual_seed(int(seed) + 7)
    return torch.randn((n_rcv, case["steps"]), generator=gen, device=dev)


def prepare(case, seed):
    dev = torch.device("cuda")
    if case["kind"] == "serve":
        jobs = []
        for k, part in enumerate(_parts(case)):
            shape = _shape(part)
            dx, dt = _grid(part)
            c, rho, cls, _, rows = _maps(part, shape, seed * 64 + k, dev)
            src, waves, wave_of, rcv = _source(part, shape, seed * 64 + k, dx, dt)
            jobs.append(dict(shape=shape, dx=dx, dt=dt, c=c, rho=rho, class_idx=cls,
                             classes=[fw.relax_params(*r[2:]) for r in rows], n_steps=case["steps"], src_mask=src,
                             waves=waves, wave_of=wave_of, rcv_mask=rcv, pml=case["pml"], f0=F0,
                             storage=case["storage"], tag=k))
        torch.cuda.synchronize()
        return dict(server=fw.Server(12 << 30), jobs=jobs)
    m, start, alpha0, n_rcv = _medium(case, seed, dev)
    dtype = torch.float64 if case["storage"] == "f64" else torch.float32
    state = dict(case=case, medium=m, start=start, traces=torch.empty((n_rcv, case["steps"]), dtype=dtype, device=dev))
    if case["kind"] == "gradient":
        state.update(alpha0=alpha0, weights=_weights(case, n_rcv, seed, dev),
                     out=tuple(torch.empty(_shape(case), device=dev) for _ in range(2)))
    else:
        state["p"] = torch.empty(_shape(case), dtype=dtype, device=dev)
    return state


def run(state):
    if "server" in state:
        server, done = state["server"], {}
        for job in state["jobs"]:
            server.submit(**job)
        while len(done) < len(state["jobs"]):
            for r in server.poll(timeout=5.0):
                if r["status"] != fw.FW_OK:
                    raise RuntimeError("request %d ended with status %d" % (r["tag"], r["status"]))
                done[r["tag"]] = r["traces"]
        return [done[k] for k in sorted(done)]
    case, m = state["case"], state["medium"]
    f64 = case["storage"] == "f64"
    m.load_state(state["start"])
    if case["kind"] == "gradient":
        gc, ga = m.gradient(case["steps"], state["weights"], alpha0=state["alpha0"], checkpoint=case["checkpoint"],
                            out=state["out"])
        return {"grad_c": gc, "grad_alpha0": ga, "traces": m.receivers(out=state["traces"])}
    m.run(case["steps"])
    return {"traces": m.receivers(f64=f64, out=state["traces"]), "p": m.read_field(fw.FW_FIELD_P, f64=f64, out=state["p"])}


# ---------------------------------------------------------------------------
# bytes and operations of one pass


def _work_forward(case):
    """Every field of the state read once and written once per step, the maps
    read once; the operations of the two half steps."""
    shape = _shape(case)
    nd, n = len(shape), float(np.prod(shape))
    es, ep = (8, 8) if case["storage"] == "f64" else (4, 2 if case["storage"] in ("bf16", "f16") else 4)
    w = case["pml"] + case["transition"]
    layer = sum(2.0 * w / s for s in shape)
    mem = 2 * (1 + nd) * es + 2 * case["mech"] * (1 + nd) * ep + 4 * layer * es
    maps = 2 * es + 2 + (es if case["nonlinear"] else 0)
    diff = 2 * nd * (11 + (12 * (nd - 1) + 10 if case["order"] == 4 else 0))
    ops = diff + nd * (9 + 5 * case["mech"]) + 8 + 5 * case["mech"] + 16 * layer
    return case["steps"] * n * (mem + maps), case["steps"] * n * ops


def work(case):
    if case["kind"] == "serve":
        each = [_work_forward(p) for p in _parts(case)]
        return {"bytes": sum(b for b, _ in each), "flops": sum(f for _, f in each)}
    b, f = _work_forward(case)
    if case["kind"] == "gradient":
        # a reverse step: the forward state of the step and the adjoint state
        # read, the adjoint state written, both gradients added to
        shape = _shape(case)
        nd, n = len(shape), float(np.prod(shape))
        state = 4 * (1 + nd) * (1 + case["mech"])
        return {"bytes": b + case["steps"] * n * (3 * state + 4 * 8 + 10),
                "flops": f + case["steps"] * n * (4 * nd * 11 + (1 + nd) * (20 + 14 * case["mech"]))}
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# the same discrete scheme in float64


def _shift(f, ax, k):
    """f at +k along ax, zero beyond the grid."""
    n = f.shape[ax]
    if k == 0:
        return f
    zero = torch.zeros_like(f.narrow(ax, 0, min(abs(k), n)))
    return torch.cat([f.narrow(ax, k, n - k), zero], ax) if k > 0 else torch.cat([zero, f.narrow(ax, 0, n + k)], ax)


def _pairs(f, ax, forward):
    """The four two-point differences of the staggered derivative along ax."""
    o = 1 if forward else 0
    return [_shift(f, ax, m + o) - _shift(f, ax, -m - 1 + o) for m in range(4)]


def _time_space(ndim):
    """Weights a_m(r^2) as polynomials: rows m, columns powers of r^2."""
    A = np.array([[(2.0 * m + 1.0) ** (2 * j + 1) for m in range(4)] for j in range(4)])
    rhs = np.eye(4)
    rhs[1:, 0] = 0.0
    rhs[:, 1] -= 2.0 * (ndim - 1) / 24.0
    return np.linalg.solve(A, rhs)


def _profile(n, w, lt, lb, off, d_top):
    x = np.arange(n) + off
    s = np.maximum(0.0, np.maximum((w - 0.5) - x, x - (n - w - 0.5)))
    if lt > 0:
        d = np.where(s <= lt, 0.1 * d_top * (s / lt) ** 2, d_top * (0.1 + 0.9 * ((s - lt) / lb) ** 2))
    else:
        d = d_top * (s / lb) ** 2
    return d * (s > 0), math.pi * F0 * (1.0 - s / w)


class _Scheme:
    """One medium in float64; scale: factor on every d of each voxel (gradients)."""

    def __init__(self, case, seed, dev, zero_state=False, grad=False):
        self.case, self.shape = case, _shape(case)
        shape, nd = self.shape, len(self.shape)
        self.nd, self.n = nd, case["mech"]
        self.dx, self.dt = _grid(case)
        c, rho, cls, beta, rows = _maps(case, shape, seed, dev)
        self.c_user = c.double().requires_grad_(grad)
        self.scale = torch.ones(shape, dtype=torch.float64, device=dev, requires_grad=True) if grad else None
        self.alpha0 = torch.tensor([r[0] for r in rows], dtype=torch.float64, device=dev)[cls.int()] if grad else None
        w = self.w = case["pml"] + case["transition"]
        at = [torch.arange(s, device=dev).clamp(w, s - 1 - w) for s in shape]

        def inherit(f):                     # the absorbing layer takes the nearest interior value
            for ax, i in enumerate(at):
                f = f.index_select(ax, i)
            return f

        c_in, self.rho, self.cls = inherit(self.c_user), inherit(rho.double()), inherit(cls.int())
        self.s_in = inherit(self.scale) if grad else None
        c_top = float(c_in.max())
        self.kdt = self.rho * c_in * c_in * self.dt
        self.b2 = 2.0 * inherit(beta.double()) * self.dt if beta is not None else None
        self.r2 = (self.kdt * self.dt / (self.rho * self.dx ** 2)) if case["order"] == 4 else None
        self.poly = _time_space(nd)
        col = lambda k, m=None: torch.tensor([r[k] if m is None else r[k][m] for r in rows], dtype=torch.float64,
                                             device=dev)
        self.kap, self.coef = [], []        # per side: kappa, [(a, b) of every mechanism]
        for kk, kd, ka in ((2, 4, 5), (3, 6, 7)):
            kap = col(kk)[self.cls]
            self.kap.append(kap)
            if grad:
                self.coef.append([self.recursion(col(kd, m)[self.cls] * self.s_in, col(ka, m)[self.cls], kap)
                                  for m in range(self.n)])
            else:
                self.coef.append([tuple(t[self.cls] for t in self.recursion(col(kd, m), col(ka, m), col(kk)))
                                  for m in range(self.n)])
        # tissue strength in the layer and the absorbing profiles per axis (array order)
        lt, lb = case["transition"], case["pml"]
        depth = torch.zeros([1] * nd, dtype=torch.float64, device=dev)
        self.absorb = []                    # per axis and side: (a, b) of the absorbing mechanism, 0 outside the layer
        d_top = -3.0 * c_top * math.log(1e-5) / (2.0 * lb * self.dx)
        for ax, s in enumerate(shape):
            view = [-1 if a == ax else 1 for a in range(nd)]
            x = torch.arange(s, dtype=torch.float64, device=dev)
            depth = torch.maximum(depth, torch.maximum(w - 0.5 - x, x - (s - w - 0.5)).clamp(min=0.0).reshape(view))
            self.absorb.append([])
            for kap, o in zip(self.kap, (0.5, 0.0)):
                d, al = (torch.from_numpy(v).to(dev).reshape(view) for v in _profile(s, w, lt, lb, o, d_top))
                a, b = self.recursion(d, al, kap)
                self.absorb[ax].append((torch.where(d > 0, a, 0.0), torch.where(d > 0, b, -1.0)))
        self.ramp = 1.0 - (depth / (lt if lt > 0 else 0.5 * lb)).clamp(max=1.0) ** 2
        z = lambda: torch.zeros(shape, dtype=torch.float64, device=dev)
        f = [z() for _ in range(1 + nd)] if zero_state else [x.double() for x in _waves(case, shape, seed, dev)]
        # state: p, v, psi1[ax][m], psi2[m], layer memory of both sides per axis (array order of axes)
        self.start = [f[0], [f[nd - ax] for ax in range(nd)], [[z() for _ in range(self.n)] for _ in range(nd)],
                      [z() for _ in range(self.n)], [z() for _ in range(nd)], [z() for _ in range(nd)]]
        src, waves, wave_of, rcv = _source(case, shape, seed, self.dx, self.dt)
        idx = lambda m: torch.from_numpy(np.flatnonzero(m)).to(dev)
        self.src, self.rcv = idx(src), idx(rcv)
        self.waves = torch.from_numpy(waves.astype(np.float64)).to(dev)[torch.from_numpy(wave_of).to(dev).long()]

    def derivative(self, f, ax, forward):
        pairs = _pairs(f, ax, forward)
        if self.r2 is None:
            cm = (1225 / 1024, -245 / 3072, 49 / 5120, -5 / 7168)
            return sum(c * p for c, p in zip(cm, pairs)) / self.dx
        r2, out = self.r2, 0.0
        for m, p in enumerate(pairs):
            q = self.poly[m]
            out = out + (((q[3] * r2 + q[2]) * r2 + q[1]) * r2 + q[0]) * p
        cross = sum(_shift(pairs[0], e, s) for e in range(self.nd) if e != ax for s in (-1, 1))
        return (out + r2 / 24.0 * cross) / self.dx

    def recursion(self, d, al, kap):
        b = torch.exp(-(d / kap + al) * self.dt)
        return d / (kap * (d + kap * al)) * (b - 1.0), b

    def stretch(self, side, g, psi):
        """Stretched derivative without the layer's mechanism, memory variables after the half step."""
        out, new, drive = g / self.kap[side], [], self.ramp * g
        for (a, b), old in zip(self.coef[side], psi):
            out = out + 0.5 * a * drive + 0.5 * (1.0 + b) * old
            new.append(b * old + a * drive)
        return out, new

    def layer(self, side, ax, g, old):
        """The absorbing mechanism along ax: its term and its memory (outside the layer the memory stays zero)."""
        a, b = self.absorb[ax][side]
        return 0.5 * (1.0 + b) * old + 0.5 * a * g, b * old + a * g

    def step(self, state, it):
        p, v, psi1, psi2, lay1, lay2 = state
        v, psi1, lay1, lay2 = list(v), list(psi1), list(lay1), list(lay2)
        for ax in range(self.nd):
            g = self.derivative(p, ax, True)
            st, psi1[ax] = self.stretch(0, g, psi1[ax])
            term, lay1[ax] = self.layer(0, ax, g, lay1[ax])
            n = self.shape[ax]
            nxt = torch.cat([self.rho.narrow(ax, 1, n - 1), self.rho.narrow(ax, n - 1, 1)], ax)
            v[ax] = v[ax] - 2.0 * self.dt / (self.rho + nxt) * (st + term)
        q = [self.derivative(v[ax], ax, False) for ax in range(self.nd)]
        div = sum(q)
        st, psi2 = self.stretch(1, div, psi2)
        for ax in range(self.nd):
            term, lay2[ax] = self.layer(1, ax, q[ax], lay2[ax])
            st = st + term
        p = p - (self.kdt if self.b2 is None else self.kdt + self.b2 * p) * st
        gain = self.kdt.reshape(-1)[self.src] / self.dx ** self.nd
        p = p.reshape(-1).index_add(0, self.src, gain * self.waves[:, it]).reshape(self.shape)
        return [p, v, psi1, psi2, lay1, lay2], p.reshape(-1)[self.rcv]

    def traces(self):
        state, cols = self.start, []
        for it in range(self.case["steps"]):
            state, col = self.step(state, it)
            cols.append(col)
        return torch.stack(cols, 1), state[0]


def _flat(state):
    p, v, psi1, psi2, l1, l2 = state
    return [p, *v, *[x for r in psi1 for x in r], *psi2, *l1, *l2]


def _unflat(f, nd, n):
    f, take = list(f), lambda k: [f.pop(0) for _ in range(k)]
    return [f.pop(0), take(nd), [take(n) for _ in range(nd)], take(n), take(nd), take(nd)]


def exact(case, seed):
    dev = torch.device("cuda")
    if case["kind"] == "serve":
        out = []
        with torch.no_grad():
            for k, part in enumerate(_parts(case)):
                out.append(_Scheme(part, seed * 64 + k, dev, zero_state=True).traces()[0].cpu().numpy())
        return out
    if case["kind"] == "forward":
        with torch.no_grad():
            tr, p = _Scheme(case, seed, dev).traces()
        return {"traces": tr, "p": p}
    # the gradient by reverse-mode differentiation, in segments recomputed from their first state
    S = _Scheme(case, seed, dev, grad=True)
    G = _weights(case, len(S.rcv), seed, dev).double()
    steps, seg = case["steps"], 8

    def span(k0, *flat):
        state, total, cols = _unflat(flat, S.nd, S.n), 0.0, []
        for it in range(k0, min(steps, k0 + seg)):
            state, col = S.step(state, it)
            cols.append(col)
            total = total + (G[:, it] * col).sum()
        return total, torch.stack(cols, 1).detach(), _flat(state)

    roots = [S.kdt, *[x for coef in S.coef for ab in coef for x in ab]]
    wrt = [x.detach().requires_grad_(True) for x in roots]
    S.kdt, rest = wrt[0], wrt[1:]
    S.coef = [[(rest[2 * (i * S.n + m)], rest[2 * (i * S.n + m) + 1]) for m in range(S.n)] for i in range(2)]
    flat, starts, cols = _flat(S.start), [], []
    with torch.no_grad():
        for k0 in range(0, steps, seg):
            starts.append(flat)
            _, col, flat = span(k0, *flat)
            cols.append(col)
    lam = [torch.zeros_like(x) for x in flat]
    acc = [torch.zeros_like(x) for x in wrt]
    for k0 in reversed(range(0, steps, seg)):
        ins = [x.detach().requires_grad_(True) for x in starts[k0 // seg]]
        total, _, outs = span(k0, *ins)
        gr = torch.autograd.grad([total, *outs], [*ins, *wrt], [torch.ones_like(total), *lam], allow_unused=True)
        lam = [torch.zeros_like(x) if g is None else g for x, g in zip(ins, gr)]
        acc = [a if g is None else a + g for a, g in zip(acc, gr[len(ins):])]
    gc, gs = torch.autograd.grad(roots, [S.c_user, S.scale], acc)
    return {"grad_c": gc, "grad_alpha0": gs / S.alpha0, "traces": torch.cat(cols, 1)}
