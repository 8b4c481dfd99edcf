"""Performance cases of the ensemble integrator: what its users have it do.

Every case goes through the package's public entry points (System, Batch,
EnsembleRK4).  The sizes are those of the package's own workloads
(wc_4k, lorenz_4M, lorenz_bif_8M, hh3_1M, mixed_batch256), of its tests and of
its benchmark, from the smallest interactive frame to ensembles that fill the
GPU, odd particle counts included.

Kinds:
  step     states in, n RK4 steps, states out (simulation without drawing);
           options: compensated update, the paper's in-kernel reset
  frames   a live view: per frame a parameter change, n steps and the density image
  grad     one training step through the integrator: loss of the end states,
           gradients of every initial state and of the parameters
  batch    many systems of all families stepped together
  sprites  soft sprites and the density image of a given state
"""
import math

import numpy as np
import torch

import paper_1505_00344_gb300 as ff
from paper_1505_00344_gb300.autograd import EnsembleRK4

# System constants (the paper's example systems at the package's workload values).
WC = [16.0, 12.0, 15.0, 3.0, 1.25, 0.0, 1.0, 1.0, 1.0, 4.0]
LORENZ = [10.0, 28.0, 8.0 / 3.0]
HH3 = [1.0, 120.0, 36.0, 0.3, 50.0, -77.0, -54.4, 0.5, -80.0, 8.0, 12.0, 10.0, 0.1, 10.0, 0.5, -20.0]
SYSTEMS = {
    "wilson_cowan": dict(params=WC, dim=2, dt=0.01, lo=[0.0] * 2, hi=[1.0] * 2),
    "lorenz": dict(params=LORENZ, dim=3, dt=0.001, lo=[-30.0, -30.0, 0.0], hi=[30.0, 30.0, 60.0]),
    "hh3": dict(params=HH3, dim=15, dt=0.01, lo=[-80.0, 0.0, 0.0, 0.0, 0.0] * 3, hi=[40.0, 1.0, 1.0, 1.0, 1.0] * 3),
}
# Floating-point operations of one particle's RK4 step as the equations are written
# (an exponential, a logarithm or a division counted as one).
FLOPS = {"wilson_cowan": 122, "lorenz": 71, "hh3": 1180}


def listed():
    return [
        # the wc_4k workload: one planar system, half its particles backward in time; the smallest
        # ensemble of the package, bound by the latency of a step
        dict(name="wc_4k", kind="step", system="wilson_cowan", particles=4096, backward=0.5, steps=1000,
             kahan=False, reset=False),
        # a phase portrait dense enough for a full-screen image
        dict(name="wc_2M", kind="step", system="wilson_cowan", particles=2_097_153, backward=0.5, steps=200,
             kahan=False, reset=False),
        # the same with the paper's particle reset: outside the unit square, or older than T_max
        dict(name="wc_reset_1M", kind="step", system="wilson_cowan", particles=1_000_000, backward=0.5, steps=200,
             kahan=False, reset=True),
        # a slider being dragged: few particles, a handful of steps per frame, so launches count
        dict(name="lorenz_live_16k", kind="frames", system="lorenz", particles=16_384, backward=0.25, steps=5,
             frames=8, width=640, height=360, bifurcation=False, kahan=False),
        # one frame of the lorenz_4M workload
        dict(name="lorenz_frame_4M", kind="frames", system="lorenz", particles=4_194_304, backward=0.25, steps=200,
             frames=1, width=1920, height=1080, bifurcation=False, kahan=False),
        # a live bifurcation diagram (r per particle), an odd count
        dict(name="lorenz_bif_2M", kind="frames", system="lorenz", particles=2_000_003, backward=0.0, steps=100,
             frames=2, width=2048, height=1024, bifurcation=True, kahan=False),
        # one small network of spiking neurons, too few particles to fill the GPU
        dict(name="hh3_12k", kind="step", system="hh3", particles=12_345, backward=0.0, steps=200, kahan=False,
             reset=False),
        # the hh3_1M workload's ensemble over a part of its run
        dict(name="hh3_1M", kind="step", system="hh3", particles=1_048_576, backward=0.0, steps=200, kahan=False,
             reset=False),
        # fitting initial states and parameters through the integrator
        dict(name="lorenz_grad_1M", kind="grad", system="lorenz", particles=1_048_576, backward=0.0, steps=400,
             every=100),
        # the same for the neurons, over a horizon at which single-precision gradients of spiking
        # trajectories still carry five digits
        dict(name="hh3_grad_64k", kind="grad", system="hh3", particles=65_537, backward=0.0, steps=60, every=30),
        # an ensemble of different models, as mixed_batch256 at a tenth of its members
        dict(name="batch_24", kind="batch", systems=24, smallest=1024, largest=524_288, steps=100, tuned=True),
        # the paper's rendering: soft sprites over the forward group of lorenz_4M
        dict(name="sprites_4M", kind="sprites", system="lorenz", particles=4_194_304, backward=0.25, radius=1.5,
             width=1920, height=1080),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _capped(rng, lo, hi, cost, most):
    """A log-uniform particle count in lo..hi whose cost per particle stays within `most`."""
    return _log(rng, lo, max(lo, min(hi, int(most / cost))))


def draw(rng):
    kind = rng.choice(["step", "step", "frames", "frames", "grad", "batch", "sprites"])
    if kind == "step":
        system = rng.choice(["wilson_cowan", "hh3", "lorenz"])
        backward = 0.0 if system == "hh3" else rng.choice([0.0, 0.25, 0.5])
        # backward in time Lorenz trajectories run off to infinity within a time unit
        steps = _log(rng, 20, 200 if system == "hh3" or (system == "lorenz" and backward) else 1000)
        most = {"wilson_cowan": 4.0e8, "hh3": 1.5e8, "lorenz": 1.2e9}[system]
        return dict(kind="step", system=system, particles=_capped(rng, 1000, 4_200_000, steps, most),
                    backward=backward, steps=steps,
                    kahan=system == "lorenz" and rng.random() < 0.3, reset=system != "hh3" and rng.random() < 0.3)
    if kind == "frames":
        frames, backward = rng.randint(1, 12), rng.choice([0.0, 0.25, 0.5])
        steps = _log(rng, 1, 200 // frames if backward else 200)
        return dict(kind="frames", system="lorenz", particles=_capped(rng, 1000, 4_200_000, frames * steps, 1.0e9),
                    backward=backward, steps=steps, frames=frames,
                    width=rng.randint(200, 2048), height=rng.randint(150, 1080), bifurcation=rng.random() < 0.4,
                    kahan=rng.random() < 0.2)
    if kind == "grad":
        system = rng.choice(["wilson_cowan", "lorenz", "hh3"])
        backward = 0.0 if system == "hh3" else rng.choice([0.0, 0.25])
        steps = _log(rng, 20, 60 if system == "hh3" else 200 if backward else 400)
        most = {"wilson_cowan": 1.0e8, "lorenz": 3.0e8, "hh3": 1.0e7}[system]
        return dict(kind="grad", system=system, particles=_capped(rng, 500, 1_100_000, steps, most),
                    backward=backward, steps=steps,
                    every=rng.choice([10, 16, 25, 50, 100]))
    if kind == "batch":
        return dict(kind="batch", systems=rng.randint(3, 30), smallest=_log(rng, 300, 3000),
                    largest=_log(rng, 10_000, 200_000), steps=_log(rng, 10, 100), tuned=rng.random() < 0.5)
    radius = round(math.exp(rng.uniform(math.log(0.75), math.log(12.0))), 2)
    return dict(kind="sprites", system=rng.choice(["lorenz", "hh3"]),
                particles=_capped(rng, 3000, 4_200_000, radius * radius + 1.0, 1.3e7), backward=rng.choice([0.0, 0.25]),
                radius=radius, width=rng.randint(200, 1920), height=rng.randint(150, 1080))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _groups(case):
    """(count, direction) of the forward and the backward group."""
    n = case["particles"]
    back = int(round(n * case["backward"]))
    return [(c, d) for c, d in ((n - back, +1), (back, -1)) if c > 0]


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(n, lo, hi, gen):
    lo, hi = (torch.tensor(v, device="cuda").reshape(-1, 1) for v in (lo, hi))
    return lo + (hi - lo) * torch.rand((lo.numel(), n), generator=gen, device="cuda")


def _params(system, seed):
    """The system's constants, the drive parameters moved a little by the seed."""
    p = list(SYSTEMS[system]["params"])
    u = np.random.default_rng(seed).uniform(-1.0, 1.0, 3)
    if system == "wilson_cowan":
        p[4] += 0.1 * u[0]
    elif system == "lorenz":
        p[1] += u[0]
    else:
        p[9:12] = [float(a + b) for a, b in zip(p[9:12], u)]
    return p


def _system(case, seed, kahan=False):
    spec = SYSTEMS[case["system"]]
    s = ff.System(case["system"], _params(case["system"], seed), case["particles"], kahan=kahan,
                  stream=torch.cuda.current_stream().cuda_stream)
    for g, (count, direction) in enumerate(_groups(case)):
        s.seed(count, spec["lo"], spec["hi"], direction, seed + 256 * g)
    return s


def _batch_members(case, seed):
    """(system, particles) of each member: types in turn, counts log-uniform (the same for every seed)."""
    sizes = np.exp(np.random.default_rng(77).uniform(math.log(case["smallest"]), math.log(case["largest"]),
                                                     case["systems"]))
    return [(("wilson_cowan", "lorenz", "hh3")[k % 3], int(round(n))) for k, n in enumerate(sizes)]


def _attractor(case, seed):
    """States to draw: around a fixed point's wings (Lorenz), anywhere in the box (the neurons)."""
    gen = _generator(seed)
    n = case["particles"]
    if case["system"] == "hh3":
        return _uniform(n, SYSTEMS["hh3"]["lo"], SYSTEMS["hh3"]["hi"], gen)
    t = torch.rand((3, n), generator=gen, device="cuda")
    side = torch.where(t[0] < 0.5, -1.0, 1.0)
    phase, rad = 2 * math.pi * t[1], 2.0 + 11.0 * torch.sqrt(t[2])
    x = side * (8.5 + 0.55 * rad * torch.cos(phase))
    y = x + side * 0.4 * rad * torch.sin(phase)
    z = 27.0 + 1.3 * rad * torch.sin(phase + 0.6)
    return torch.stack([x, y, z])


def _camera(width, height):
    """Column-major model-view-projection of a pinhole camera at (150, 150, 150) looking at (-20, -20, -20)."""
    eye, at, up = (np.array(v, float) for v in ((150.0,) * 3, (-20.0,) * 3, (0.0, 0.0, 1.0)))
    f = (at - eye) / np.linalg.norm(at - eye)
    s = np.cross(f, up)
    s /= np.linalg.norm(s)
    view = np.eye(4)
    view[:3, :3] = np.stack([s, np.cross(s, f), -f])
    view[:3, 3] = -view[:3, :3] @ eye
    t = 1.0 / math.tan(math.radians(45.0) / 2)
    proj = np.zeros((4, 4))
    proj[0, 0], proj[1, 1], proj[3, 2] = t * height / width, t, -1.0
    proj[2, 2], proj[2, 3] = (1000.0 + 1.0) / (1.0 - 1000.0), 2 * 1000.0 / (1.0 - 1000.0)
    return (proj @ view).T.reshape(16).astype(np.float32)


def _view(case):
    w, h = case["width"], case["height"]
    if case["system"] == "hh3":
        return dict(ndim_view=3, axes=(0, 5, 10), mvp=_camera(w, h), width=w, height=h)
    if case.get("bifurcation"):
        return dict(ndim_view=2, axes=(3, 2), lo=(0.0, 0.0), hi=(200.0, 400.0), width=w, height=h)
    return dict(ndim_view=2, axes=(0, 2), lo=(-30.0, 0.0), hi=(30.0, 60.0), width=w, height=h)


def _sprite(case):
    return dict(radius=case["radius"], gain=0.75, colours=[[1.0, 0.8, 0.4, 1.0], [0.2, 0.4, 1.0, 1.0]])


def _frame_params(case, seed):
    """The parameters before each frame: the r (bifurcation: beta) slider moving."""
    p = _params("lorenz", seed)
    out = []
    for f in range(case["frames"]):
        q = list(p)
        q[2 if case["bifurcation"] else 1] += 0.1 * f
        out.append(q)
    return out


def prepare(case, seed):
    gen = _generator(seed)
    kind = case["kind"]
    if kind == "batch":
        members = _batch_members(case, seed)
        systems, x0 = [], []
        for k, (name, n) in enumerate(members):
            one = dict(system=name, particles=n, backward=0.0)
            systems.append(_system(one, seed + 1000 * k))
            x0.append(_uniform(n, SYSTEMS[name]["lo"], SYSTEMS[name]["hi"], gen))
        batch = ff.Batch(systems, torch.cuda.current_stream().cuda_stream)
        dts = [SYSTEMS[name]["dt"] for name, _ in members]
        if case["tuned"]:
            batch.autotune(dts, 16)
        return dict(case=case, batch=batch, systems=systems, x0=x0, dts=dts, out=[torch.empty_like(x) for x in x0])
    spec = SYSTEMS[case["system"]]
    s = _system(case, seed, kahan=case.get("kahan", False))
    st = dict(case=case, system=s, dt=spec["dt"])
    if kind == "step":
        st["x0"] = _uniform(case["particles"], spec["lo"], spec["hi"], gen)
        st["out"] = torch.empty_like(st["x0"])
        if case["reset"]:
            lo, hi, t_max, every = ([0.0] * 2, [1.0] * 2, 5.0, 1) if case["system"] == "wilson_cowan" else \
                                   ([-60.0, -60.0, -20.0], [60.0, 60.0, 100.0], 0.0, 10)
            s.set_reset(lo, hi, t_max, every)
            st["age"], st["resets"] = (torch.zeros(case["particles"], dtype=torch.int32, device="cuda") for _ in "ab")
    elif kind == "frames":
        if case["bifurcation"]:
            s.set_particle_param(1, 0.0, 200.0)
        st["params"] = _frame_params(case, seed)
        st["view"] = ff.make_view(**_view(case))
        st["images"] = torch.zeros((case["frames"], case["height"], case["width"]), dtype=torch.int32, device="cuda")
        st["out"] = torch.empty((3, case["particles"]), device="cuda")
    elif kind == "grad":
        st["x0"] = _uniform(case["particles"], spec["lo"], spec["hi"], gen).requires_grad_()
        st["target"] = _uniform(case["particles"], spec["lo"], spec["hi"], gen)
        st["params"] = torch.tensor(_params(case["system"], seed), dtype=torch.float32, requires_grad=True)
    else:
        s.set_state(_attractor(case, seed))
        st["view"], st["sprite"] = ff.make_view(**_view(case)), ff.make_sprite(**_sprite(case))
        st["counts"] = torch.zeros((case["height"], case["width"]), dtype=torch.int32, device="cuda")
        st["colours"] = torch.zeros((case["height"], case["width"], 4), device="cuda")
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "batch":
        for s, x in zip(st["systems"], st["x0"]):
            s.set_state(x)
        st["batch"].step(case["steps"], st["dts"])
        for s, o in zip(st["systems"], st["out"]):
            s.get_state(o)
        return st["out"]
    s = st["system"]
    if kind == "step":
        s.set_state(st["x0"])
        s.step(case["steps"], st["dt"])
        s.get_state(st["out"])
        if not case["reset"]:
            return dict(state=st["out"])
        s.get_reset_state(st["age"], st["resets"])
        return dict(state=st["out"], age=st["age"], resets=st["resets"])
    if kind == "frames":
        s.reset()
        for f, p in enumerate(st["params"]):
            s.set_params(p)
            s.step_splat(case["steps"], st["dt"], st["view"], st["images"][f])
        s.get_state(st["out"])
        return dict(state=st["out"], images=st["images"])
    if kind == "grad":
        end = EnsembleRK4.apply(st["x0"], st["params"], s, case["steps"], st["dt"], case["every"])
        loss = ((end - st["target"]) ** 2).sum() / case["particles"]
        dx0, dp = torch.autograd.grad(loss, (st["x0"], st["params"]))
        return dict(end=end.detach(), dx0=dx0, dp=dp)
    s.project_splat(st["view"], st["counts"])
    s.project_sprites(st["view"], st["sprite"], st["colours"])
    return dict(counts=st["counts"], colours=st["colours"])


def work(case):
    kind = case["kind"]
    if kind == "batch":
        m = _batch_members(case, 0)
        return dict(bytes=sum(8.0 * SYSTEMS[s]["dim"] * n for s, n in m),
                    flops=sum(float(FLOPS[s]) * n for s, n in m) * case["steps"])
    n, d = case["particles"], SYSTEMS[case["system"]]["dim"]
    if kind == "step":
        return dict(bytes=n * (8.0 * d + (8.0 if case["reset"] else 0.0)),
                    flops=float(FLOPS[case["system"]]) * n * case["steps"])
    if kind == "frames":
        # the states (made from the seed) written once, each frame's image written once
        return dict(bytes=n * (4.0 * d + (4.0 if case["bifurcation"] else 0.0))
                    + 4.0 * case["frames"] * case["width"] * case["height"],
                    flops=float(FLOPS["lorenz"]) * n * case["steps"] * case["frames"])
    if kind == "grad":
        # initial states and targets read, end states and gradients written; a reverse step is
        # four vector-Jacobian products, about twice a step's operations, after the forward step
        return dict(bytes=16.0 * d * n, flops=3.0 * FLOPS[case["system"]] * n * case["steps"])
    # the drawn coordinates read by both techniques, both images written; per covered pixel its
    # distance (6), falloff (3) and four channels (8)
    axes = 3 if case["system"] == "hh3" else 2
    return dict(bytes=4.0 * axes * n + 20.0 * case["width"] * case["height"],
                flops=17.0 * math.pi * case["radius"] ** 2 * n)


# ---------------------------------------------------------------------------
# The same in 64 bits, plain torch
# ---------------------------------------------------------------------------
def _rhs_wc(x, p):
    E, I = x
    S = lambda a: 1.0 / (1.0 + torch.exp(-p[8] * (a - p[9])))  # noqa: E731
    return [(-E + S(p[0] * E - p[1] * I + p[4])) / p[6], (-I + S(p[2] * E - p[3] * I + p[5])) / p[7]]


def _rhs_lorenz(x, p):
    return [p[0] * (x[1] - x[0]), x[0] * (p[1] - x[2]) - x[1], x[0] * x[1] - p[2] * x[2]]


def _rate(v):
    """v / (1 - exp(-v / 10)), 10 at v = 0."""
    small = v.abs() < 1e-9
    safe = torch.where(small, torch.ones_like(v), v)
    return torch.where(small, 10.0 + v / 2, safe / -torch.expm1(-safe / 10.0))


def _rhs_hh3(x, p):
    C, gNa, gK, gL, ENa, EK, EL, gsyn, Esyn, I1, I2, I3, tr, td, sig, theta = p
    total = x[4] + x[9] + x[14]
    out = []
    for i, drive in enumerate((I1, I2, I3)):
        V, m, h, n, s = x[5 * i:5 * i + 5]
        am, bm = 0.1 * _rate(V + 40.0), 4.0 * torch.exp(-(V + 65.0) / 18.0)
        ah, bh = 0.07 * torch.exp(-(V + 65.0) / 20.0), 1.0 / (1.0 + torch.exp(-(V + 35.0) / 10.0))
        an, bn = 0.01 * _rate(V + 55.0), 0.125 * torch.exp(-(V + 65.0) / 80.0)
        act = 1.0 / (1.0 + torch.exp(-sig * (V - theta)))
        dV = (drive + gNa * m ** 3 * h * (ENa - V) + gK * n ** 4 * (EK - V) + gL * (EL - V)
              + gsyn * (total - s) * (Esyn - V)) / C
        out += [dV, am * (1 - m) - bm * m, ah * (1 - h) - bh * h, an * (1 - n) - bn * n, act * (1 - s) / tr - s / td]
    return out


RHS = {"wilson_cowan": _rhs_wc, "lorenz": _rhs_lorenz, "hh3": _rhs_hh3}


def _rk4(name, x, p, h):
    f = lambda y: torch.stack(RHS[name](list(y.unbind(0)), p))  # noqa: E731
    k1 = f(x)
    k2 = f(x + 0.5 * h * k1)
    k3 = f(x + 0.5 * h * k2)
    k4 = f(x + h * k3)
    return x + h / 6.0 * (k1 + 2.0 * k2 + 2.0 * k3 + k4)


def _signed_dt(case):
    dt = SYSTEMS[case["system"]]["dt"]
    return torch.cat([torch.full((c,), d * dt, dtype=torch.float64, device="cuda") for c, d in _groups(case)])


def _splitmix_seed(case, seed):
    """The groups' initial states: draw n = j * dim + k + 1 of the SplitMix64 stream, its top 24 bits."""
    spec = SYSTEMS[case["system"]]
    d, parts = spec["dim"], []
    lo, hi = np.array(spec["lo"]), np.array(spec["hi"])
    with np.errstate(over="ignore"):
        for g, (count, _) in enumerate(_groups(case)):
            z = np.uint64(seed + 256 * g) + np.arange(1, count * d + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
            u = ((z ^ (z >> np.uint64(31))) >> np.uint64(40)).astype(np.float64) / 2.0 ** 24
            parts.append((lo + (hi - lo) * u.reshape(count, d)).astype(np.float32).T)
    return torch.from_numpy(np.ascontiguousarray(np.concatenate(parts, axis=1))).cuda().double()


def _exact_grad(case, seed):
    spec, gen = SYSTEMS[case["system"]], _generator(seed)
    x = _uniform(case["particles"], spec["lo"], spec["hi"], gen).double()
    target = _uniform(case["particles"], spec["lo"], spec["hi"], gen).double()
    p = torch.tensor(_params(case["system"], seed), dtype=torch.float32).double().cuda().requires_grad_()
    h = _signed_dt(case)
    states = []
    with torch.no_grad():
        for _ in range(case["steps"]):
            states.append(x)
            x = _rk4(case["system"], x, p, h)
    end, lam, dp = x, 2.0 * (x - target) / case["particles"], torch.zeros_like(p)
    for x in reversed(states):
        x = x.detach().requires_grad_()
        lam, q = torch.autograd.grad(_rk4(case["system"], x, p, h), (x, p), lam)
        dp = dp + q
    return dict(end=end, dx0=lam, dp=dp.detach())


def _exact_sprites(case, seed):
    x = _attractor(case, seed).double()
    w, h, R = case["width"], case["height"], case["radius"]
    if case["system"] == "hh3":
        m = torch.from_numpy(_camera(w, h)).cuda().double().reshape(4, 4)
        clip = torch.stack([x[0], x[5], x[10], torch.ones_like(x[0])], 1) @ m
        keep = clip[:, 3] > 0
        col = (clip[:, 0] / clip[:, 3] + 1.0) * (w / 2)
        row = (clip[:, 1] / clip[:, 3] + 1.0) * (h / 2)
    else:
        keep = torch.ones_like(x[0], dtype=torch.bool)
        col, row = (x[0] + 30.0) * (w / 60.0), x[2] * (h / 60.0)
    spec = _sprite(case)
    group = torch.cat([torch.full((c,), g, device="cuda") for g, (c, _) in enumerate(_groups(case))])
    colour = spec["gain"] * torch.tensor(spec["colours"], dtype=torch.float64, device="cuda")
    planes = torch.zeros((2, h * w), dtype=torch.float64, device="cuda")
    reach = int(math.ceil(R)) + 1
    c0, r0 = torch.floor(col).long(), torch.floor(row).long()
    for dr in range(-reach, reach + 1):
        for dc in range(-reach, reach + 1):
            c, r = c0 + dc, r0 + dr
            q = ((c + 0.5 - col) ** 2 + (r + 0.5 - row) ** 2) / (float(np.float32(R)) ** 2)
            on = keep & (q < 1.0) & (c >= 0) & (c < w) & (r >= 0) & (r < h)
            planes.view(-1).index_add_(0, ((group * h + r) * w + c)[on], ((1.0 - q) ** 2)[on])
    return dict(counts=None, colours=torch.einsum("gp,gk->pk", planes, colour[:2]).reshape(h, w, 4))


def exact(case, seed):
    kind = case["kind"]
    if kind == "grad":
        return _exact_grad(case, seed)
    if kind == "sprites":
        return _exact_sprites(case, seed)
    with torch.no_grad():
        if kind == "batch":
            gen, out = _generator(seed), []
            for k, (name, n) in enumerate(_batch_members(case, seed)):
                x = _uniform(n, SYSTEMS[name]["lo"], SYSTEMS[name]["hi"], gen).double()
                for _ in range(case["steps"]):
                    x = _rk4(name, x, _params(name, seed + 1000 * k), SYSTEMS[name]["dt"])
                out.append(x)
            return out
        h = _signed_dt(case)
        if kind == "step":
            if case["reset"]:  # where a particle is re-drawn hangs on single roundings: no value in 64 bits
                return None
            spec = SYSTEMS[case["system"]]
            x = _uniform(case["particles"], spec["lo"], spec["hi"], _generator(seed)).double()
            p = _params(case["system"], seed)
            for _ in range(case["steps"]):
                x = _rk4(case["system"], x, p, h)
            return dict(state=x)
        x = _splitmix_seed(case, seed)
        n = case["particles"]
        r = 200.0 * torch.arange(n, dtype=torch.float64, device="cuda") / max(1, n - 1)
        for p in _frame_params(case, seed):
            if case["bifurcation"]:
                p = [p[0], r.float().double(), p[2]]
            for _ in range(case["steps"]):
                x = _rk4("lorenz", x, p, h)
        return dict(state=x, images=None)
