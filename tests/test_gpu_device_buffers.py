"""Device buffers given by their address, whose size the binding cannot check, and calls that fail."""
import pytest

torch = pytest.importorskip("torch")

import paper_1505_00344_gb300 as ff  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ff.lib()


def test_a_reported_error_does_not_fail_the_next_call():
    """A call that a CUDA error ends (here an allocation far beyond the memory) leaves nothing behind that
    the next call's launch check would report once more."""
    s = ff.System("lorenz", [10.0, 28.0, 8 / 3], 100, stream=torch.cuda.current_stream().cuda_stream)
    with pytest.raises(ff.FFError):
        ff.System("lorenz", [10.0, 28.0, 8 / 3], 10 ** 12, stream=torch.cuda.current_stream().cuda_stream)
    s.seed(100, [-30, -30, 0], [30, 30, 60], 1, 3)
    s.step(1, 0.001)
