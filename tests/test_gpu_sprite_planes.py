"""Sprites through weight planes (FF_SPRITE_AUTO with enough particles for the image's size, from
a system's second such picture on) against the direct technique."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1505_00344_gb300 as ff  # noqa: E402

pytestmark = pytest.mark.gpu
BOX = ([-30, -30, 0], [30, 30, 60])


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ff.lib()


def lorenz(counts, stream=None):
    s = ff.System("lorenz", [10.0, 28.0, 8 / 3], sum(counts), stream=stream or torch.cuda.current_stream().cuda_stream)
    for g, c in enumerate(counts):
        s.seed(c, *BOX, 1, 70 + g)
    return s


def view(width, height, **more):
    # the particles fill the middle half of the window in x and z
    return dict(dict(ndim_view=2, axes=(0, 2), lo=(-60.0, -30.0), hi=(60.0, 90.0), width=width, height=height), **more)


def draw(s, v, sprite, image):
    s.project_sprites(v, sprite, image)
    torch.cuda.synchronize()
    return image.cpu().numpy()


def ready(s):
    """The system's first picture that asks for the planes is drawn directly; the next ones use them."""
    img = torch.zeros((10, 10, 4), device="cuda")
    s.project_sprites(view(10, 10), dict(radius=12.0, colours=[[1.0] * 4] * 8), img)


@pytest.mark.parametrize("accumulate", [0, 1])
def test_a_colour_that_overflows_stays_on_the_pixels_its_sprites_cover(accumulate):
    """gain and colour are finite, their product is not: pixels a sprite of that group covers become
    infinite (weight times infinity), all others keep what the other groups give them, and none is NaN --
    on both techniques, which cover the same pixels."""
    s = lorenz([3000, 40, 3000])
    ready(s)
    colours = [[1.0, 0.0, 0.5, 1.0], [3e38, 0.25, 0.0, 3e38], [0.0, 0.3, 0.9, 0.125]]
    out = []
    for technique in (ff.FF_SPRITE_AUTO, ff.FF_SPRITE_DIRECT):
        img = torch.full((95, 161, 4), 0.5 if accumulate else 7.0, device="cuda")
        out.append(draw(s, view(161, 95, accumulate=accumulate),
                        dict(radius=12.0, gain=2.0, colours=colours, technique=technique), img))
    got, want = out
    assert np.isinf(want).any() and np.isfinite(want).any() and not np.isnan(want).any()
    np.testing.assert_array_equal(np.isinf(got), np.isinf(want))
    assert not np.isnan(got).any()
    m = np.isfinite(want)
    # at most 6,040 fragments a pixel: the two orders of FP32 additions differ by less than 2 (f + 8) 2^-24
    np.testing.assert_allclose(got[m], want[m], rtol=2 * 6048 * 2.0 ** -24, atol=0)


def test_pictures_leave_another_streams_capture_alone():
    """A picture that allocates or grows the workspace, drawn while another stream captures in the
    strictest mode (which refuses calls that may synchronise, and is lost by one): the picture is the direct
    technique's and the captured graph replays to the steps' states."""
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    a, b, called = lorenz([3000, 3000], mine.cuda_stream), lorenz([3000], other.cuda_stream), lorenz([3000])
    ready(a)
    sprite = dict(radius=12.0, gain=0.5, colours=[[1.0, 0.5, 0.25, 1.0]] * 8)
    sizes = [(160, 96), (320, 180)]
    images = [torch.zeros((h, w, 4), device="cuda") for w, h in sizes]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(other):
        graph.capture_begin(capture_error_mode="global")
        try:
            b.step(3, 0.001)
            for (w, h), img in zip(sizes, images):
                a.project_sprites(view(w, h), sprite, img)
        finally:
            graph.capture_end()
        graph.replay()
    called.step(3, 0.001)
    torch.cuda.synchronize()
    x, y = np.empty((3, 3000), np.float32), np.empty((3, 3000), np.float32)
    b.get_state(x)
    called.get_state(y)
    np.testing.assert_array_equal(x, y)
    for (w, h), img in zip(sizes, images):
        want = draw(a, view(w, h), dict(sprite, technique=ff.FF_SPRITE_DIRECT), torch.zeros_like(img))
        np.testing.assert_allclose(img.cpu().numpy(), want, rtol=2 * 6008 * 2.0 ** -24, atol=0)
