"""Sprites through weight planes (FF_SPRITE_AUTO with enough particles for the image's size, once
the system's pictures could have saved what the workspace costs) against the oracle and the direct technique."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
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


def ready(s, width, height):
    """Pictures of that size until by the size rule the system holds planes for it and all its groups."""
    saving = s.info()[0] * (np.pi * 32 * 32 - 32.5 ** 2) - 0.2 * 3 * width * height - 1e6
    img = torch.zeros((height, width, 4), device="cuda")
    for _ in range(1 + int(2e7 / saving)):
        s.project_sprites(view(width, height), dict(radius=32.0, colours=[[1.0] * 4] * 8), img)


@pytest.mark.parametrize("accumulate", [0, 1])
def test_a_colour_that_overflows_stays_on_the_pixels_its_sprites_cover(accumulate):
    """gain and colour are finite, their product is not: pixels a sprite of that group covers become
    infinite (weight times infinity), all others keep what the other groups give them, and none is NaN --
    on both techniques, which cover the same pixels."""
    s = lorenz([3000, 40, 3000])
    ready(s, 161, 95)
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


PICTURES = [(160, 96, 12.0, 0b111, 0), (37, 25, 12.0, 0b111, 0), (161, 95, 20.0, 0b101, 0), (160, 96, 16.0, 0b010, 1),
            (64, 201, 32.0, 0b111, 1), (1, 1, 32.0, 0b111, 0), (2, 3, 14.5, 0b110, 1), (640, 361, 32.0, 0b001, 0),
            (160, 96, 12.0, 0b111, 0)]


def test_one_system_draws_pictures_of_many_sizes():
    """Sizes, radii and group masks change from picture to picture on one system, whose workspace serves
    them all: every picture is the oracle's of that view alone, each channel within (f + 8) 2^-24 of
    the sum of its f fragments' magnitudes (f additions and the rounding of each contribution), untouched
    pixels exactly as they were."""
    counts = [2300, 1900, 2100]
    s = lorenz(counts)
    ready(s, 640, 361)
    n, group = sum(counts), np.repeat(np.arange(3, dtype=np.int32), counts)
    x = np.empty((3, n), np.float32)
    s.get_state(x)
    colours = [[1.0, 0.25, 0.0, 1.0], [0.0, 0.5, 1.0, -0.75], [0.3, -1.0, 0.6, 2.0]]
    rng = np.random.default_rng(2)
    for W, H, R, mask, accumulate in PICTURES:
        drawn = bin(mask).count("1")
        assert n * (np.pi * R * R - (R + 0.5) ** 2) > 0.2 * drawn * W * H + 1e6  # the planes' size rule
        v = view(W, H, group_mask=mask, accumulate=accumulate)
        base = rng.uniform(-1, 1, (H, W, 4)).astype(np.float32)
        got = draw(s, v, dict(radius=R, gain=0.8, colours=colours), torch.from_numpy(base).cuda()).astype(np.float64)
        want, absum, frags = oracle.sprites2d(x[0], x[2], v["lo"], v["hi"], W, H, R, 0.8, colours, group=group,
                                              include=((mask >> group) & 1).astype(np.uint8))
        base = base * float(accumulate)
        assert (np.abs(got - base - want) <= (frags[:, :, None] + 8.0) * 2.0 ** -24 * (absum + np.abs(base))).all()
        np.testing.assert_array_equal(got[frags == 0], base[frags == 0])


@pytest.mark.parametrize("radius", [0.95, 1.5])
def test_small_sprites_of_many_particles_match_the_oracle(radius):
    """As above for sprites of one to a few pixels, of which it takes many to pay for the planes."""
    counts = [1_500_000, 5, 1_500_000]
    s = lorenz(counts)
    ready(s, 400, 301)
    n, group = sum(counts), np.repeat(np.arange(3, dtype=np.int32), counts)
    assert n * (np.pi * radius ** 2 - (radius + 0.5) ** 2) > 0.2 * 3 * 400 * 301 + 1e6
    x = np.empty((3, n), np.float32)
    s.get_state(x)
    colours, v = [[1.0, 0.25, 0.0, 1.0], [0.0, 0.5, 1.0, -0.75], [0.3, -1.0, 0.6, 2.0]], view(400, 301)
    got = draw(s, v, dict(radius=radius, gain=0.8, colours=colours), torch.zeros((301, 400, 4), device="cuda"))
    want, absum, frags = oracle.sprites2d(x[0], x[2], v["lo"], v["hi"], 400, 301, radius, 0.8, colours, group=group)
    assert (np.abs(got.astype(np.float64) - want) <= (frags[:, :, None] + 8.0) * 2.0 ** -24 * absum).all()
    np.testing.assert_array_equal(got[frags == 0], 0.0)


def test_pictures_leave_another_streams_capture_alone():
    """A picture that allocates or grows the workspace, drawn while another stream captures in the
    strictest mode (which refuses calls that may synchronise, and is lost by one): the picture is the direct
    technique's and the captured graph replays to the steps' states."""
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    a, b, called = lorenz([6000, 6000], mine.cuda_stream), lorenz([3000], other.cuda_stream), lorenz([3000])
    sprite = dict(radius=32.0, gain=0.5, colours=[[1.0, 0.5, 0.25, 1.0]] * 8)
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
        np.testing.assert_allclose(img.cpu().numpy(), want, rtol=2 * 12008 * 2.0 ** -24, atol=0)


@pytest.mark.parametrize("n,radius,pictures,allocates", [(400_000, 1.5, 3, False), (400_000, 12.0, 1, True)])
def test_the_workspace_comes_once_it_would_have_paid(n, radius, pictures, allocates):
    """A system whose pictures save little draws several of them without the workspace (16 bytes a pixel
    block of 4096 x 2160, 35 MB); one whose first picture saves more than the allocation costs has it at once."""
    s = lorenz([n])
    img = torch.zeros((400, 400, 4), device="cuda")
    big = torch.zeros((2160, 4096, 4), device="cuda")

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    if not allocates:
        assert 0 < n * (np.pi * radius ** 2 - (radius + 0.5) ** 2) - 0.2 * 400 * 400 - 1e6 < 2e7 / pictures
    # (the direct kernel's first launch loads its code)
    s.project_sprites(view(400, 400), dict(radius=1.0, colours=[[1.0] * 4] * 8, technique=ff.FF_SPRITE_DIRECT), img)
    before = free()
    for _ in range(pictures):
        s.project_sprites(view(*((4096, 2160) if allocates else (400, 400))), dict(radius=radius, colours=[[1.0] * 4] * 8),
                          big if allocates else img)
    assert (before - free() >= 30 * 2 ** 20) == allocates
    assert allocates or before == free()
