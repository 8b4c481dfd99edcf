"""Calls that a size rule sends to another kernel, or whose launch the caller shapes, against the
general path: the same bits and no less of the GPU."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1505_00344_gb300 as ff  # noqa: E402

pytestmark = pytest.mark.gpu
WC = [16.0, 12.0, 15.0, 3.0, 1.25, 0.0, 1.0, 1.0, 1.0, 4.0]
HH = [1.0, 120.0, 36.0, 0.3, 50.0, -77.0, -54.4, 0.5, -80.0, 8.0, 12.0, 10.0, 0.1, 10.0, 0.5, -20.0]
BOX = {"wilson_cowan": ([0, 0], [1, 1]), "lorenz": ([-30, -30, 0], [30, 30, 60]),
       "hh3": ([-80.0, 0, 0, 0, 0] * 3, [40.0, 1, 1, 1, 1] * 3)}
PARAMS = {"wilson_cowan": WC, "lorenz": [10.0, 28.0, 8 / 3], "hh3": HH}


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ff.lib()


def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def system(name, *counts, params=None):
    """A forward group of the first count and, where given, a backward and another forward one."""
    s = ff.System(name, params or PARAMS[name], sum(counts), stream=torch.cuda.current_stream().cuda_stream)
    for g, c in enumerate(counts):
        s.seed(c, *BOX[name], -1 if g == 1 else 1, 40 + g)
    return s


def states(s):
    n, _, dim, _ = s.info()
    x = np.empty((dim, n), np.float32)
    s.get_state(x)
    return x


# Wilson-Cowan's packed pairs: groups of even and odd counts that start on even and odd particles, a
# small group before and after a large one.
@pytest.mark.parametrize("small", [(), (1,), (1000,), (1001, 7)])
@pytest.mark.parametrize("first", [0, 5])
def test_wilson_cowan_pairs_keep_the_one_particle_bits(small, first):
    """The pairs' states are the one-particle kernel's to the bit: untaped and taped, alone and in a batch,
    in the unit square, where a logistic is far below 2^-60 (|E|, |I| up to 20 and a steep slope), at
    zero, and at infinite and NaN states (NaN for NaN)."""
    counts = ((first,) if first else ()) + (650 * sms() + 3,) + small
    n = sum(counts)
    rng = np.random.default_rng(4)
    wide = rng.uniform(-20, 20, (2, n)).astype(np.float32)
    odd = np.array([np.nan, np.inf, -np.inf, 3e38, -3e38, 1e-30, -0.0, 0.0, 1.0], np.float32)
    wide[:, :81] = np.array(np.meshgrid(odd, odd)).reshape(2, -1)
    for params, x0 in ((WC, None), (WC, wide), (WC[:8] + [9.0, 2.0], wide)):
        out = []
        for form in ("pairs", "one", "taped", "batched"):
            s = system("wilson_cowan", *counts, params=params)
            if x0 is not None:
                s.set_state(x0)
            if form == "one":
                s.set_launch(1)
            if form == "taped":
                s.tape_begin(3, 7)
            if form == "batched":
                b = ff.Batch([s], torch.cuda.current_stream().cuda_stream)
                b.step(7, [0.01])
            else:
                s.step(7, 0.01)
            if form == "pairs":
                assert "wc_rk4_x2u" in s.last_launch()["kernel"]
            out.append(states(s))
        for x in out[1:]:
            np.testing.assert_array_equal(out[0], x)


# The launch of the default shape where particles reset, or where sigma or beta is taken per particle,
# in the range where two particles per thread at 16 warps per SM run otherwise.
@pytest.mark.parametrize("form", ["reset", "reset, r each", "sigma each", "beta each"])
def test_default_lorenz_shape_of_other_kernels_fills_the_gpu(form):
    """The one-block shape belongs to the group-uniform packed kernel: every other launch has the grid and
    block that a caller gets who asks for four particles per thread, and the same states."""
    n = 3000 * sms() + 5
    out = []
    for ppt in (0, 4):
        s = system("lorenz", 4 * (n // 8), n - 4 * (n // 8))
        s.set_launch(ppt)
        if form != "reset":
            s.set_particle_param({"reset, r each": 1, "sigma each": 0, "beta each": 2}[form], 2.0, 12.0)
        if "reset" in form:
            s.set_reset([-20, -25, 2], [20, 25, 45], 0.02, 1)
        s.step(9, 0.004)
        out.append((s.last_launch(), states(s)))
    np.testing.assert_array_equal(out[0][1], out[1][1])
    a, b = out[0][0], out[1][0]
    assert (a["grid"], a["block"]) == (b["grid"], b["block"])


# Resetting pairs with several rounds of work per warp, Lorenz at the default shape's ranges.
@pytest.mark.parametrize("name,per_sm", [("lorenz", 150), ("lorenz", 3000), ("lorenz", 9000), ("wilson_cowan", 6000)])
def test_large_resetting_ensembles_match_their_parts(name, per_sm):
    """An ensemble's states, ages and reset counts are those of its slices of up to 1,000 particles per SM
    run alone, bit for bit."""
    n, lim = per_sm * sms() + 3, {"lorenz": ([-20, -25, 2], [20, 25, 45]),
                                  "wilson_cowan": ([0.1, 0.05], [0.9, 0.95])}[name]

    def run(first, count):
        s = ff.System(name, PARAMS[name], count, stream=torch.cuda.current_stream().cuda_stream)
        s.seed_slice(count, first, n, *BOX[name], 1, 40)
        s.set_reset(*lim, 0.05, 2)
        s.step(21, 0.01)
        age, res = (np.empty(count, np.uint32) for _ in "ab")
        s.get_reset_state(age, res)
        return np.concatenate([states(s).view(np.uint32), age[None], res[None]])

    whole, part = run(0, n), 1000 * sms() + 1
    for first in range(0, n, part):
        np.testing.assert_array_equal(run(first, min(part, n - first)), whole[:, first:first + part])


# A caller's limit of blocks per SM, which counts blocks of the block size it goes with.
@pytest.mark.parametrize("name,n,blocks,block,reset", [
    ("hh3", 12_345, 1, 0, False), ("hh3", 25_001, 2, 96, False), ("hh3", 50_000, 1, 128, False),
    ("lorenz", 400_001, 1, 0, True), ("wilson_cowan", 400_001, 1, 512, True), ("wilson_cowan", 400_001, 1, 512, False),
    ("wilson_cowan", 400_001, 3, 0, False), ("wilson_cowan", 400_001, 1, 1024, True)])
def test_a_limit_of_blocks_per_sm_keeps_its_threads(name, n, blocks, block, reset):
    """Whatever kernel runs, it has as many threads per SM as the caller's limit gives (blocks times the block
    size, at most the 512 or 256 of the system's one-particle kernel), if it has the work, and no more."""
    s = system(name, n)
    s.set_launch(0, block, blocks)
    if reset:
        s.set_reset([v - 1 for v in BOX[name][0]], [v + 1 for v in BOX[name][1]], 0.0, 1)
    s.step(2, 0.001)
    launch = s.last_launch()
    most = 256 if name == "hh3" else 512
    size = min(block or (512 if name == "lorenz" else 256), most)
    limit = blocks * size * sms()
    pairs, lanes = ("x2" in launch["kernel"] or "pair" in launch["kernel"]), "lane_integrate" in launch["kernel"]
    work = (n + 19) // 20 * 32 if lanes else ((n + 1) // 2 if pairs else n)  # lanes: up to 20 particles a warp
    threads = launch["grid"] * launch["block"]
    assert min(limit, work) <= threads <= max(limit, work + launch["block"] - 1), launch
