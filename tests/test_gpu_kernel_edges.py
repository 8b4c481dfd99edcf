"""Kernels and dispatch rules at the sizes where they can go wrong: edges of tiles and
blocks, remainders, the smallest and largest of their ranges."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1505_00344_gb300 as ff  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ff.lib()


def _stream():
    return torch.cuda.current_stream().cuda_stream


# The parameter gradient's partial rows (one per 128-particle block here): one row, one less
# than, as many as and more than the summing block's 128 threads, and several rounds of them.
@pytest.mark.parametrize("n", [1, 127 * 128, 128 * 128, 128 * 128 + 1, 700 * 128 + 37])
def test_parameter_gradient_sums_every_partial_row(n):
    """dL/dp of an ensemble is the sum of its slices' dL/dp.  The per-particle contributions
    are the same FP32 values, so only the order of FP64 additions differs: n + 2 roundings of
    at most sum |c| each, far below 1e-9 of it (here contributions of one sign dominate)."""
    def grad(first, count):
        s = ff.System("harmonic", [1.3], count, stream=_stream())
        s.seed_slice(count, first, n, [0.5, -1.0], [1.0, 1.0], +1, 91)
        s.tape_begin(8, 16)
        s.step(16, 0.05)
        lam = torch.ones((2, count), device="cuda")
        return s.backward(lam, lam, 1)[0]

    cuts = [0, n // 3, n] if n >= 3 else [0, n]
    parts = sum(grad(a, b - a) for a, b in zip(cuts, cuts[1:]))
    whole = grad(0, n)
    assert abs(whole - parts) <= 1e-9 * abs(whole)


# Boxes at the edges of the pair arithmetic of the draws: ordinary ones, intervals far from
# zero, across zero, of width zero, much narrower than their offset, at and beyond the scales
# that take the double formula, and bounds that are no floats.
BOXES = [(0.0, 1.0), (-30.0, 30.0), (-80.0, 40.0), (0.1, 0.30000000000000004), (1e6, 1e6 + 1e-3), (-1e-3, 1e6),
         (3.0, 3.0), (0.0, 0.0), (-0.0, 1e-11), (-1e-13, 1e-13), (2.0**-42, 2.0**-41), (-1e30, 1e30), (-1e31, 2e31),
         (-3e38, 3e38), (1.0, 1.0 + 2.0**-23), (-1.0 / 3.0, 2.0 / 3.0)]


@pytest.mark.parametrize("count", [1, 257, 40_003])
def test_seeding_is_the_double_formula_for_every_box(count):
    """x = fl32(lo + width * u), both double operations rounded, for u the top 24 bits of
    SplitMix64 output j * dim + k + 1 -- bit for bit, whichever arithmetic formed it."""
    with np.errstate(over="ignore"):
        z = np.uint64(99) + np.arange(1, 2 * count + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        u = ((z ^ (z >> np.uint64(31))) >> np.uint64(40)).astype(np.float64) / 2.0 ** 24
    u = u.reshape(count, 2).T
    for a, b in zip(BOXES[0::2], BOXES[1::2]):
        lo, hi = np.array([[a[0]], [b[0]]]), np.array([[a[1]], [b[1]]])
        with np.errstate(over="ignore"):
            want = (lo + (hi - lo) * u).astype(np.float32)
        s = ff.System("harmonic", [1.0], count, stream=_stream())
        s.seed(count, [a[0], b[0]], [a[1], b[1]], +1, 99)
        got = np.empty((2, count), np.float32)
        s.get_state(got)
        np.testing.assert_array_equal(got.view(np.uint32), want.view(np.uint32), err_msg=f"{a} {b}")


HH = [1.0, 120.0, 36.0, 0.3, 50.0, -77.0, -54.4, 0.5, -80.0, 8.0, 12.0, 10.0, 0.1, 10.0, 0.5, -20.0]
HH_BOX = ([-80.0, 0.0, 0.0, 0.0, 0.0] * 3, [40.0, 1.0, 1.0, 1.0, 1.0] * 3)


# HH x 3 at two particles per thread picks its kernel by size: a partial, full and just
# overfull warp of 10 and of 20 particles, and either side of the lines between kernels.
@pytest.mark.parametrize("n", [1, 3, 9, 10, 11, 21, -1, -2, -3, -4, -5, -6])
@pytest.mark.parametrize("variant", ["plain", "parameter", "taped"])
def test_hh3_kernels_by_size_give_the_one_particle_bits(n, variant):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = {-1: 120 * sms, -2: 120 * sms + 1, -3: 400 * sms, -4: 400 * sms + 1, -5: 256 * sms, -6: 256 * sms + 1}.get(n, n)
    out = []
    for ppt in (1, 2):
        s = ff.System("hh3", HH, n, stream=_stream())
        back = n // 3  # a group boundary inside a pair where it is odd
        s.seed(n - back, *HH_BOX, +1, 5)
        if back:
            s.seed(back, *HH_BOX, -1, 6)
        s.set_launch(ppt)
        if variant == "parameter":
            s.set_particle_param(9, 5.0, 15.0)
        if variant == "taped":
            s.tape_begin(3, 8)
        s.step(7, 0.01)
        x = np.empty((15, n), np.float32)
        s.get_state(x)
        out.append(x)
        if variant == "taped":
            lam = torch.ones((15, n), device="cuda")
            s.backward(lam, lam, 16)
            out[-1] = np.concatenate([x, lam.cpu().numpy()])
    np.testing.assert_array_equal(out[0], out[1])


WC = [16.0, 12.0, 15.0, 3.0, 1.25, 0.0, 1.0, 1.0, 1.0, 4.0]


def _wc(n, back, ppt, seed=11, first=None, total=None):
    s = ff.System("wilson_cowan", WC, n, stream=_stream())
    if total is None:
        s.seed(n - back, [0, 0], [1, 1], +1, seed)
        if back:
            s.seed(back, [0, 0], [1, 1], -1, seed + 1)
    else:
        s.seed_slice(n, first, total, [0, 0], [1, 1], +1, seed)
    s.set_launch(ppt)
    return s


def _states(s):
    n, _, dim, _ = s.info()
    x = np.empty((dim, n), np.float32)
    s.get_state(x)
    return x


# Wilson-Cowan at two particles per thread: either side of the line between its kernels, odd
# counts, a second group that starts inside a pair, a small group beside a large one.
@pytest.mark.parametrize("extra,back,kernel", [(0, 0, "wc_rk4_x2u"), (-1, 0, "integrate_kernel"), (1000, 1000, "wc_rk4_x2u"),
                                               (1002, 1001, "wc_rk4_x2u"), (1, 1, "wc_rk4_x2u"), (500, 1000, "integrate_kernel")])
def test_wilson_cowan_pairs_by_size(extra, back, kernel):
    """The packed pairs against an FP64 RK4: each step rounds a state below 1.5 (1.5 backward)
    by at most an ulp or two of it and the errors grow with the map, at most e^3.2 (the largest
    eigenvalue of the reversed flow, 3.2, over one time unit) backward: 100 steps stay within
    1e-5 of max(|x|, 1), the package's bar for this system."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 650 * sms + extra
    s = _wc(n, back, 0)
    x = torch.from_numpy(_states(s)).cuda().double()
    h = torch.full((n,), 0.01, dtype=torch.float64, device="cuda")
    h[n - back:] *= -1.0 if back else 1.0
    s.step(100, 0.01)
    assert kernel in s.last_launch()["kernel"]

    def f(E, I):
        S = lambda a: 1.0 / (1.0 + torch.exp(-WC[8] * (a - WC[9])))  # noqa: E731
        return torch.stack([-E + S(WC[0] * E - WC[1] * I + WC[4]), -I + S(WC[2] * E - WC[3] * I + WC[5])])

    for _ in range(100):
        k1 = f(*x)
        k2 = f(*(x + 0.5 * h * k1))
        k3 = f(*(x + 0.5 * h * k2))
        k4 = f(*(x + h * k3))
        x = x + h / 6 * (k1 + 2 * k2 + 2 * k3 + k4)
    want = x.cpu().numpy()
    assert (np.abs(_states(s) - want) / np.maximum(np.abs(want), 1.0)).max() <= 1e-5


def test_wilson_cowan_slices_and_odd_values_match_the_whole():
    """A slice of an ensemble takes its whole ensemble's kernel: the slices' states are the
    whole's to the bit.  Infinite and NaN states give the one-particle kernel's."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 650 * sms
    whole = _wc(n, 0, 0, first=0, total=n)
    whole.step(50, 0.01)
    for a, b in ((0, 10), (10, 4001), (4001, n)):
        part = _wc(b - a, 0, 0, first=a, total=n)
        part.step(50, 0.01)
        np.testing.assert_array_equal(_states(part), _states(whole)[:, a:b])
    # pieces beside each other that start and end inside a pair, and beside a small group
    part = ff.System("wilson_cowan", WC, 17, stream=_stream())
    part.seed_slice(5, 0, n, [0, 0], [1, 1], +1, 11)
    part.seed(7, [0, 0], [1, 1], +1, 12)
    part.seed_slice(5, 5, n, [0, 0], [1, 1], +1, 11)
    part.step(50, 0.01)
    got = _states(part)
    np.testing.assert_array_equal(np.concatenate([got[:, :5], got[:, 12:]], axis=1), _states(whole)[:, :10])
    small = _wc(7, 0, 1, seed=12)
    small.step(50, 0.01)
    np.testing.assert_array_equal(got[:, 5:12], _states(small))
    odd = np.array([np.nan, np.inf, -np.inf, 3e38, -3e38, 1e30, 0.0, 1.0], np.float32)
    x0 = np.tile(np.array(np.meshgrid(odd, odd)).reshape(2, -1), n // 64 + 1)[:, :n].copy()
    got = []
    for ppt in (1, 2):
        s = _wc(n, 0, ppt)
        s.set_state(x0)
        s.step(3, 0.01)
        got.append(_states(s))
    np.testing.assert_array_equal(np.isfinite(got[0]), np.isfinite(got[1]))
    np.testing.assert_array_equal(np.isnan(got[0]), np.isnan(got[1]))


# Particle reset in packed pairs: single particles, odd and even totals and a second group,
# against one-particle launches (an odd first group keeps those).
@pytest.mark.parametrize("counts", [(1,), (2,), (1, 5), (64, 3), (4098, 2001), (4097, 2000)])
@pytest.mark.parametrize("system", ["wilson_cowan", "lorenz"])
@pytest.mark.parametrize("bounds,t_max,every", [(True, 0.0, 1), (False, 0.07, 1), (True, 0.11, 3)])
def test_reset_pairs_match_particles_alone(counts, system, bounds, t_max, every):
    """The same ensemble with each group's first particle cut off into a system of its own
    (a slice, so it draws as itself): every state, age and count agrees bit for bit with the
    ensemble cut after an even and after an odd particle, which swaps lanes and kernels."""
    params, box, lim, dt = {
        "wilson_cowan": (WC, ([0, 0], [1, 1]), ([0.1, 0.05], [0.9, 0.95]), 0.01),
        "lorenz": ([10.0, 28.0, 8 / 3], ([-30, -30, 0], [30, 30, 60]), ([-20, -25, 2], [20, 25, 45]), 0.01)}[system]
    dim = len(box[0])

    def run(parts):
        s = ff.System(system, params, sum(n for _, _, n, _ in parts), stream=_stream())
        for g, first, n, total in parts:
            s.seed_slice(n, first, total, *box, 1 if g == 0 else -1, 40 + g)
        s.set_reset(*(lim if bounds else (None, None)), t_max, every)
        s.step(13, dt)
        s.step(20, dt)
        x = _states(s)
        age, res = (np.empty(x.shape[1], np.uint32) for _ in "ab")
        s.get_reset_state(age, res)
        return np.concatenate([x.view(np.uint32), age[None], res[None]])

    whole = run([(g, 0, n, n) for g, n in enumerate(counts)])
    start = 0
    for g, n in enumerate(counts):
        cut = min(n, 1 + 2 * (n // 5))  # odd: the second part's pairs are the whole's shifted by one
        parts = [run([(g, 0, cut, n)])] + ([run([(g, cut, n - cut, n)])] if n > cut else [])
        np.testing.assert_array_equal(np.concatenate(parts, axis=1), whole[:, start:start + n])
        start += n


# Sprites through weight planes: odd and even images, one pixel, a sprite larger than the image,
# a masked group in front, both view kinds, clearing and accumulating, a host image.
@pytest.mark.parametrize("width,height,radius", [(1, 1, 1.5), (2, 3, 0.8), (37, 25, 4.0), (64, 48, 32.0), (33, 70, 1.5)])
@pytest.mark.parametrize("mask,accumulate,host", [(0xFFFFFFFF, 0, False), (0b10, 1, False), (0b101, 1, True)])
def test_sprite_planes_match_the_direct_technique(width, height, radius, mask, accumulate, host):
    """Both techniques cover the same pixels with the same weights and differ in the order of
    FP32 additions: |difference| <= 2 (f + 8) 2^-24 sum |c| of a pixel with f fragments, and
    here at most n fragments of at most 0.9 each meet (untouched pixels agree exactly)."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 1_200_000 if radius > 1.0 else 9_000_000  # beyond the line between the techniques
    counts = [n // 3, 5, n - n // 3 - 5]
    s = ff.System("lorenz", [10.0, 28.0, 8 / 3], n, stream=_stream())
    for g, c in enumerate(counts):
        s.seed(c, [-30, -30, 0], [30, 30, 60], 1, 70 + g)
    view = dict(ndim_view=2, axes=(0, 2), lo=(-28.0, 1.0), hi=(29.0, 57.0), width=width, height=height,
                group_mask=mask, accumulate=accumulate)
    colours = [[1.0, 0.0, 0.5, 1.0], [0.25, 1.0, 1.0, 0.0], [0.0, 0.3, 0.9, 0.125]]
    base = torch.linspace(0, 1, width * height * 4, device="cuda").reshape(height, width, 4)
    out = []
    for technique in (ff.FF_SPRITE_AUTO, ff.FF_SPRITE_DIRECT):
        img = base.cpu().numpy().copy() if host else base.clone()
        if technique == ff.FF_SPRITE_AUTO:  # a system's first picture is a direct one; the planes are clear after each
            for _ in range(2):
                scratch = torch.zeros_like(base)
                s.project_sprites(dict(view, accumulate=0), dict(radius=radius, colours=colours), scratch)
        for _ in range(2 if not accumulate else 1):
            s.project_sprites(view, dict(radius=radius, gain=0.9, colours=colours, technique=technique), img)
        out.append(img if host else img.cpu().numpy())
    fragments = np.abs(out[1] - (base.cpu().numpy() if accumulate else 0)).max() / (0.9 * 0.125) + 1
    bar = 2 * (min(n, 60 * fragments) + 8) * 2.0 ** -24 * (np.abs(out[1]) + 1.0)
    assert (np.abs(out[0] - out[1]) <= bar).all()
    assert np.array_equal(out[0][out[1] == (base.cpu().numpy() if accumulate else 0)],
                          out[1][out[1] == (base.cpu().numpy() if accumulate else 0)])


# Device copies of the state: runs of 4,096, planes at every offset modulo 16 bytes, an unaligned
# base, a buffer the copy kernel may not touch (pinned host memory given by its address).
@pytest.mark.parametrize("n", [1, 2, 3, 5, 255, 4095, 4096, 4097, 8192, 12290])
@pytest.mark.parametrize("dim,offset", [(2, 0), (3, 1), (15, 2), (15, 3)])
def test_device_state_copies(n, dim, offset):
    rhs, params = {2: ("harmonic", [1.0]), 3: ("lorenz", [10.0, 28.0, 8 / 3]), 15: ("hh3", HH)}[dim]
    s = ff.System(rhs, params, n, stream=_stream())
    s.seed(n, [0.0] * dim, [1.0] * dim, 1, 3)
    want = _states(s)
    buf = torch.full((dim * n + 8,), -7.0, device="cuda")
    s.get_state(buf[offset:offset + dim * n])
    got = buf.cpu().numpy()
    np.testing.assert_array_equal(got[offset:offset + dim * n].reshape(dim, n), want)
    assert (got[:offset] == -7).all() and (got[offset + dim * n:] == -7).all()
    new = torch.rand(dim * n + 8, device="cuda")
    s.set_state(new[offset:offset + dim * n])
    np.testing.assert_array_equal(_states(s), new[offset:offset + dim * n].cpu().numpy().reshape(dim, n))
    pinned = torch.zeros(dim * n).pin_memory()
    ff.ff_get_state(s.handle, pinned.data_ptr())
    torch.cuda.synchronize()
    np.testing.assert_array_equal(pinned.numpy().reshape(dim, n), _states(s))


# Batch tiles by the batch's size: members of one particle and of odd counts, beside one large
# enough that tiles grow to several items a thread, at the default and at tuned shapes.
@pytest.mark.parametrize("counts", [(1, 2, 5), (63, 130, 4097), (7, 300_003, 900)])
@pytest.mark.parametrize("tuned", [False, True])
def test_batch_tiles_cover_every_particle(counts, tuned):
    def members():
        out = []
        for q, n in enumerate(counts):
            for name, p, box in (("hh3", HH, HH_BOX), ("wilson_cowan", WC, ([0, 0], [1, 1]))):
                s = ff.System(name, p, n, stream=_stream())
                s.seed(n, *box, +1, 50 + q)
                out.append(s)
        return out

    batched, alone = members(), members()
    dts = [0.01] * len(batched)
    b = ff.Batch(batched, _stream())
    if tuned:
        b.autotune(dts, 2)
    b.step(4, dts)
    for x, y in zip(batched, alone):
        y.set_launch(1)
        y.step(4, 0.01)
        np.testing.assert_array_equal(_states(x), _states(y))


@pytest.mark.parametrize("n", [25, 130_003])
def test_handed_out_work_replays_and_is_deterministic(n):
    """The queue that hands out a launch's tasks is clear for the next one: a captured step
    replays to the states of the calls, and two sweeps of one tape give the same gradients."""
    side = torch.cuda.Stream()
    captured, called = (ff.System("hh3", HH, n, stream=side.cuda_stream) for _ in "ab")
    for s in (captured, called):
        s.seed(n, *HH_BOX, +1, 5)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        captured.step(3, 0.01)
    for _ in range(3):
        with torch.cuda.stream(side):
            graph.replay()
        called.step(3, 0.01)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(_states(captured), _states(called))
    for rhs, params, box, every in (("lorenz", [10.0, 28.0, 8 / 3], ([-30, -30, 0], [30, 30, 60]), 20),
                                    ("lorenz", [10.0, 28.0, 8 / 3], ([-30, -30, 0], [30, 30, 60]), 10),
                                    ("hh3", HH, HH_BOX, 10)):
        dim = len(box[0])
        s = ff.System(rhs, params, n, stream=_stream())
        s.seed(n, *box, +1, 5)
        s.tape_begin(every, 40)
        s.step(40, 0.001)
        lam = torch.randn((dim, n), device="cuda")
        got = []
        for _ in range(2):
            out = torch.empty_like(lam)
            got.append((s.backward(lam, out, len(params)).copy(), out))
        np.testing.assert_array_equal(got[0][0], got[1][0])
        assert torch.equal(got[0][1], got[1][1])


# The default Lorenz shape by size: either side of each line, groups that start on even and odd
# particles, with and without a parameter per particle, against four particles per thread.
@pytest.mark.parametrize("per_sm,extra", [(200, -1), (200, 0), (2500, -1), (2500, 3), (5000, 1), (20000, 0)])
@pytest.mark.parametrize("odd,parameter", [(0, False), (1, False), (2, True)])
def test_default_lorenz_shape_keeps_the_bits(per_sm, extra, odd, parameter):
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + extra
    first = n // 2 // 4 * 4 + odd
    view = dict(ndim_view=2, axes=(0, 2), lo=(-30.0, 0.0), hi=(30.0, 60.0), width=320, height=180)
    out = []
    for ppt in (0, 4):
        s = ff.System("lorenz", [10.0, 28.0, 8 / 3], n, stream=_stream())
        s.seed(first, [-30, -30, 0], [30, 30, 60], +1, 5)
        s.seed(n - first, [-30, -30, 0], [30, 30, 60], -1, 6)
        if parameter:
            s.set_particle_param(1, 20.0, 40.0)
        s.set_launch(ppt)
        img = torch.zeros((180, 320), dtype=torch.int32, device="cuda")
        s.step_splat(7, 0.001, view, img)
        s.step(5, 0.001)
        out.append((_states(s), img.cpu().numpy()))
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("n", [1, 63, 130, 20_001])
def test_lorenz_sweep_uniform_and_general_agree(n):
    """One group with one set of parameters takes the uniform sweep; the same particles as two
    groups take the general one: the same operations in the same tasks, so the same bits."""
    def grads(groups):
        s = ff.System("lorenz", [10.0, 28.0, 8 / 3], n, stream=_stream())
        first = 0
        for c in groups:
            s.seed_slice(c, first, n, [-30, -30, 0], [30, 30, 60], +1, 5)
            first += c
        s.tape_begin(33, 100)
        s.step(100, 0.001)
        out = torch.empty_like(lam)
        return s.backward(lam, out, 3).copy(), out.cpu().numpy()

    lam = torch.randn((3, n), device="cuda", generator=torch.Generator(device="cuda").manual_seed(3))
    one = grads([n])
    two = grads([n // 3, n - n // 3] if n > 2 else [n])
    np.testing.assert_array_equal(one[1], two[1])
    np.testing.assert_array_equal(one[0], two[0])
