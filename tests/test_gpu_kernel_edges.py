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
