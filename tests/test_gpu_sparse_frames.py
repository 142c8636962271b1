"""Frames in which most regions hold no or few records (needs a GB300): what is written where
nothing is drawn, for rows of every alignment, and that such frames take no longer than their
neighbours in size."""
import statistics

import numpy as np
import pytest
import torch

import oracle
import oracle_pins as P
from paper_1606_04427_gb300 import build, render

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    assert torch.cuda.is_available()


def _set(W, H, n, R, seed=0, part=1.0):
    rng = np.random.default_rng(seed)
    s = 2.0 / P.focal(H)
    px, py = rng.uniform(0.5 - 0.5 * part, 0.5 + 0.5 * part, (2, n)) * np.array([[W], [H]])
    return P.make_set(0.5 + (px - 0.5 * W) * s, 0.5 - (py - 0.5 * H) * s, np.full(n, 0.5), np.full(n, R / 0.75 * s),
                      rng.uniform(0.0, 1.0, n), beta=0.5)


# a pixel sums at most n terms in FP32; a term's own error is below 4e-6 (as in the tests of teams)
@pytest.mark.parametrize("W", [96, 97, 98, 100])
@pytest.mark.parametrize("n,R", [(1, 2.5), (12, 5.0), (150, 2.0)])
def test_every_pixel_is_written(W, n, R):
    H = 75
    ps = _set(W, H, n, R, n)
    cam = P.front(W, H)
    a = oracle.render(ps, cam)
    sc = render.Scene(ps, "f32")
    held = torch.linspace(-1.0, 3.0, H * W * 3, device="cuda").reshape(H, W, 3)
    for T in (5, 16, 20, 24, 40, 64):
        for mode, want in (("", oracle.final(a)), ("accum", a), ("add", held.cpu().numpy() + a)):
            out = held.clone() if mode == "add" else torch.full((H, W, 3), float("nan"), device="cuda")
            got = sc.render(cam, render.RenderParams(tile=T, accum=mode == "accum", add=mode == "add"), out)
            np.testing.assert_allclose(got.cpu().numpy(), want, rtol=n * 2.0 ** -24 + 4e-6,
                                       atol=4 * 2.0 ** -24 if mode == "add" else 1e-12, err_msg=f"T={T} {mode}")
            untouched = a == 0
            assert np.array_equal(got.cpu().numpy()[untouched], (want if mode != "add" else held.cpu().numpy())[untouched])


def _ms(sc, cam, out):
    times = []
    for _ in range(30):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        sc.render(cam, None, out)
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b))
    return statistics.median(times[5:])


def _frame_ms(W, n, part=1.0):
    sc, out = render.Scene(_set(W, W, n, 0.1, 1, part), "f16"), torch.empty(W, W, 3, device="cuda")
    return _ms(sc, P.front(W, W), out)


def test_rows_of_any_alignment_take_the_same_time():
    """A width that is not a multiple of four is written value by value: the splat of 10 k particles
    took 0.19 ms at 4095^2 where it took 0.12 at 4096^2 (the frame about 1.35 times as long)."""
    assert _frame_ms(4095, 10_000) < 1.2 * _frame_ms(4096, 10_000)


def test_regions_of_14_pixels_take_no_longer_per_pixel():
    """Nor are the rows of regions of 14 pixels aligned: per pixel, a frame of 10 k particles took 1.4
    times as long at 5000^2 (tiles of 40) as at 4096^2 (tiles of 32)."""
    assert _frame_ms(5000, 10_000) / 5000 ** 2 < 1.2 * _frame_ms(4096, 10_000) / 4096 ** 2


def test_more_particles_are_not_faster():
    """Lists of 300 records in tiles of 24 pixels: shared by teams of four, whose parts then hold a few
    records of a region, 1 M particles took 1.4 times as long as 1.2 M in teams of two."""
    assert _frame_ms(2501, 1_000_000, 0.6) < 1.15 * _frame_ms(2501, 1_200_000, 0.6)
