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


def _states(s):
    n, _, dim, _ = s.info()
    x = np.empty((dim, n), np.float32)
    s.get_state(x)
    return x


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
