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
