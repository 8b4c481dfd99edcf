"""Device buffers given by their address, whose size the binding cannot check, and calls that fail."""
import ctypes

import pytest

torch = pytest.importorskip("torch")

import paper_1505_00344_gb300 as ff  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ff.lib()


def captured(call, stream):
    """The types of the nodes (0 kernel, 1 copy) that the call adds to a captured graph, which is never
    launched, or None if the call is refused."""
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    refused = False
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        graph.capture_begin(capture_error_mode="relaxed")
        try:
            call()
        except ff.FFError:
            refused = True
        try:
            graph.capture_end()
        except RuntimeError:
            assert refused
    if refused:
        return None
    cuda, handle = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p(graph.raw_cuda_graph())
    n, types = ctypes.c_size_t(8), []
    nodes = (ctypes.c_void_p * 8)()
    assert cuda.cuGraphGetNodes(handle, nodes, ctypes.byref(n)) == 0
    for node in nodes[:n.value]:
        kind = ctypes.c_int(-1)
        assert cuda.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        types.append(kind.value)
    return types


def test_the_copy_kernel_keeps_within_the_callers_allocation():
    """A buffer that ends before the state does is left to the copy call, which checks its ranges and
    refused it before; the copy kernel, which would access what lies beyond, takes whole buffers only.
    (Seen in captured graphs: nothing is copied here.)"""
    stream = torch.cuda.Stream()
    n = 8_000_003  # 96 MB; the allocator rounds the small buffer up to 2 MB
    s = ff.System("lorenz", [10.0, 28.0, 8 / 3], n, stream=stream.cuda_stream)
    s.seed(n, [-30, -30, 0], [30, 30, 60], 1, 3)
    small, whole = torch.zeros(64, device="cuda"), torch.zeros(3 * n, device="cuda")
    for f in (ff.ff_get_state, ff.ff_set_state):
        assert captured(lambda: f(s.handle, whole.data_ptr()), stream) == [0]
        for address in (small.data_ptr(), whole.data_ptr() + 4 * 1024 ** 2):
            nodes = captured(lambda: f(s.handle, address), stream)
            assert nodes is None or nodes == [1]


def test_a_reported_error_does_not_fail_the_next_call():
    """A call that a CUDA error ends (here an allocation far beyond the memory) leaves nothing behind that
    the next call's launch check would report once more."""
    s = ff.System("lorenz", [10.0, 28.0, 8 / 3], 100, stream=torch.cuda.current_stream().cuda_stream)
    with pytest.raises(ff.FFError):
        ff.System("lorenz", [10.0, 28.0, 8 / 3], 10 ** 12, stream=torch.cuda.current_stream().cuda_stream)
    s.seed(100, [-30, -30, 0], [30, 30, 60], 1, 3)
    s.step(1, 0.001)
