"""Frames of few records are splatted by teams of 8, 4 or 2 warps, each warp taking a consecutive
part of a long item's records; items of at most 32 records are evaluated without batches (needs
a GB300).  On 152 SMs x 16 warps and items of 2048 records the team's size changes at 1.0, 2.5
and 7.5 M records; the crowds below reach each, on few tiles and on many."""
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


def _set(W, H, crowd, spread):
    """`crowd` particles on one 16-pixel tile, `spread` over the whole image."""
    rng = np.random.default_rng(crowd + spread)
    n = crowd + spread
    px = np.concatenate([rng.uniform(96.0, 112.0, crowd), rng.uniform(0.0, W, spread)])
    py = np.concatenate([rng.uniform(32.0, 48.0, crowd), rng.uniform(0.0, H, spread)])
    R = np.concatenate([rng.uniform(0.8, 12.0, crowd), rng.uniform(0.8, 30.0, spread)])
    s = 2.0 / P.focal(H)  # world units per pixel on the plane z = 0.5
    return P.make_set(0.5 + (px - 0.5 * W) * s, 0.5 - (py - 0.5 * H) * s, np.full(n, 0.5), R / 0.75 * s,
                      rng.uniform(0.0, 1.0, n), beta=0.01)


# n non-negative FP32 terms summed in any order: (n - 1) 2^-24 relative; a term's own error is
# below 4e-6 (a weight's exponent at most 5.8, rounded five times; the exponential's 2^-22).
@pytest.mark.parametrize("crowd,spread", [(0, 1), (32, 0), (33, 40), (255, 31), (513, 300), (9001, 257)])
@pytest.mark.parametrize("tiles", [(1, 1), (39, 32), (128, 128)])
def test_teams_match_the_oracle(tiles, crowd, spread):
    W, H = 16 * tiles[0], 16 * tiles[1]
    ps = _set(W, H, crowd, spread)
    cam = P.front(W, H)
    want = oracle.render(ps, cam)
    sc = render.Scene(ps, "f32")
    rtol = (crowd + spread - 1) * 2.0 ** -24 + 4e-6
    for T in (16, 40):
        got = sc.render(cam, render.RenderParams(tile=T, accum=True)).cpu().numpy()
        np.testing.assert_allclose(got, want, rtol=rtol, atol=1e-12, err_msg=f"T={T}")
    first, again = (sc.render(cam, render.RenderParams(accum=True, stable=True)) for _ in range(2))
    assert torch.equal(first, again)


@pytest.mark.parametrize("n", [900_000, 1_100_000, 2_400_000, 2_600_000, 7_400_000, 7_600_000])
def test_team_sizes_agree(n):
    """About n records (supports of at most a pixel, one tile each or two at its edge) over 64
    tiles: teams of 8, 4, 2 and lone warps against the same sums over tiles of 8 pixels, whose
    items are other slices."""
    W = H = 128
    rng = np.random.default_rng(n)
    s = 2.0 / P.focal(H)
    px, py = rng.uniform(0.5, W - 0.5, (2, n))
    ps = P.make_set(0.5 + (px - 0.5 * W) * s, 0.5 - (py - 0.5 * H) * s, np.full(n, 0.5), np.full(n, 0.2 / 0.75 * s),
                    rng.uniform(0.0, 1.0, n), beta=0.01)
    cam = P.front(W, H)
    sc = render.Scene(ps, "f32")
    a, b = (sc.render(cam, render.RenderParams(tile=T, accum=True)).cpu().numpy() for T in (16, 8))
    # a pixel holds about n / 128^2 < 500 terms; both sums within (terms - 1) 2^-24 of the exact one
    np.testing.assert_allclose(a, b, rtol=2 * 1000 * 2.0 ** -24, atol=1e-12)
    first, again = (sc.render(cam, render.RenderParams(accum=True, stable=True)) for _ in range(2))
    assert torch.equal(first, again)


@pytest.mark.parametrize("W,H", [(64, 48), (70, 33), (45, 31)])  # rows of 16, 8 and 4 bytes' alignment
@pytest.mark.parametrize("crowd,spread", [(0, 3), (70, 200), (5001, 2000)])
def test_added_images_hold_the_sum(W, H, crowd, spread):
    """A render added into an image: every pixel is what it held plus the accumulation."""
    ps = _set(W, H, crowd, spread)
    ps.x[:crowd] -= np.float32((104.0 - 20.0) * 2.0 / P.focal(H))  # the crowd moves into the image
    cam = P.front(W, H)
    sc = render.Scene(ps, "f32")
    for T in (16, 40):
        acc = sc.render(cam, render.RenderParams(tile=T, accum=True, stable=True))
        held = torch.linspace(-1.0, 3.0, H * W * 3, device="cuda").reshape(H, W, 3)
        out = held.clone()
        sc.render(cam, render.RenderParams(tile=T, add=True, stable=True), out)
        assert torch.equal(out, held + acc)
