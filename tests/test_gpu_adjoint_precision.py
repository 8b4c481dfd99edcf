"""Precision of single gradient components of HH x 3, particle by particle: sums over many particles
average an FP32 accumulation's rounding away."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import paper_1505_00344_gb300 as ff  # noqa: E402

pytestmark = pytest.mark.gpu
HH = [1.0, 120.0, 36.0, 0.3, 50.0, -77.0, -54.4, 0.5, -80.0, 8.0, 12.0, 10.0, 0.1, 10.0, 0.5, -20.0]
BOX = ([-80.0, 0, 0, 0, 0] * 3, [40.0, 1, 1, 1, 1] * 3)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ff.lib()


@pytest.mark.parametrize("every,bar", [(100, 2.6e-6), (256, 3.9e-6)])
def test_hh3_capacitance_gradient_keeps_the_net_current(every, bar):
    """dL/dC is minus the sum over the steps of (dV/dt) v_V / C, in which large ionic currents cancel:
    summed as a net current, 128 particles one at a time have a median relative error against the
    FP64 sensitivities of 1.7e-6 over 100 steps and 2.6e-6 over 256 (a chunk each), which is mostly the
    FP32 trajectory's; the currents' separate sums, cancelled at the chunk's end, have 5.5e-6.  The
    bars are one and a half times the former."""
    total = 128
    p64 = [float(np.float32(v)) for v in HH]
    x0 = oracle.seed_group(15, *BOX, 17, count=total)
    lam = np.random.default_rng(3).standard_normal((15, total)).astype(np.float32)
    _, _, Q = oracle.tangent(oracle.HH3, x0, p64, 0.01, every)
    each = np.einsum("pi,ip->p", Q[:, :, 0], lam.astype(np.float64))
    err = []
    for i in range(total):
        s = ff.System("hh3", HH, 1, stream=torch.cuda.current_stream().cuda_stream)
        s.seed(1, *BOX, 1, 5)
        s.set_state(np.ascontiguousarray(x0[:, i:i + 1]))
        s.tape_begin(every, every)
        s.step(every, 0.01)
        v = torch.from_numpy(np.ascontiguousarray(lam[:, i:i + 1])).cuda()
        err.append(abs(s.backward(v, torch.empty_like(v), 16)[0] / each[i] - 1.0))
    assert np.median(err) <= bar, np.median(err)


def test_hh3_products_hold_beta_n_to_the_forwards_precision():
    """At n = 1 the derivative of dn/dt with respect to V is beta_n / 80 but for cancelling terms: one Euler
    step's dL/dV for L = n, over V from -82 to -70 mV where those are small.  With beta_n as the forward forms it the
    rms relative error is 5.5e-8; with its factor folded into the exponent, whose offset then has
    twice the rounding error, 9.9e-8."""
    n, h = 200_000, 0.0078125
    V = np.linspace(-82.0, -70.0, n).astype(np.float32)
    x = np.full((15, n), 0.5, np.float32)
    x[0::5], x[3::5] = V, 1.0
    s = ff.System("hh3", HH, n, method="euler", stream=torch.cuda.current_stream().cuda_stream)
    s.seed(n, *BOX, 1, 5)
    s.set_state(x)
    s.tape_begin(1, 1)
    s.step(1, h)
    lam = np.zeros((15, n), np.float32)
    lam[3::5] = 1.0
    v = torch.from_numpy(lam).cuda()
    out = torch.empty_like(v)
    s.backward(v, out, 16)
    want = h / 80.0 * 0.125 * np.exp(-(V.astype(np.float64) + 65.0) / 80.0)
    err = out.cpu().numpy()[0::5] / want - 1.0
    assert np.sqrt((err ** 2).mean()) <= 7e-8
