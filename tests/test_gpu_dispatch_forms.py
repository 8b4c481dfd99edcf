"""Calls that a size rule sends to another kernel, or whose launch the caller shapes, against the
general path: the same bits and no less of the GPU."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1505_00344_gb300 as ff  # noqa: E402

pytestmark = pytest.mark.gpu
WC = [16.0, 12.0, 15.0, 3.0, 1.25, 0.0, 1.0, 1.0, 1.0, 4.0]
BOX = {"wilson_cowan": ([0, 0], [1, 1])}
PARAMS = {"wilson_cowan": WC}



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
