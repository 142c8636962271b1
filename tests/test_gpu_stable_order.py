"""SPLOTCH_STABLE images are the same bits on every run, whichever warps and teams take which
work items (needs a GB300).  The frames here have far more items than teams of warps (304 teams of
8 on 152 SMs), so that which team meets which item changes from run to run."""
import numpy as np
import pytest
import torch

import oracle_pins as P
from paper_1606_04427_gb300 import build, render

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    assert torch.cuda.is_available()


def _scene(W, H, px, py, R, seed):
    """Particles at image positions px, py with support radius R (pixels)."""
    s = 2.0 / P.focal(H)
    n = px.shape[0]
    I = np.random.default_rng(seed).uniform(0.0, 1.0, n)
    return render.Scene(P.make_set(0.5 + (px - 0.5 * W) * s, 0.5 - (py - 0.5 * H) * s, np.full(n, 0.5),
                                   R / 0.75 * s, I, beta=0.01), "f32")


def _tiles(W, H, T, counts, margin, rng):
    """counts[k] particles on tile k (row-major), at least `margin` of its part of the image from
    that part's edges."""
    nx = -(-W // T)
    who = np.repeat(np.arange(counts.size), counts)
    out = []
    for at, size in ((who % nx * T, W), (who // nx * T, H)):
        out.append(at + rng.uniform(margin, 1.0 - margin, who.size) * np.minimum(T, size - at))
    return out


def test_short_items_do_not_depend_on_when_a_team_parts():
    """Thousands of lists of 33 to 64 records behind a few long ones: every team parts at one of
    them, and other such items go to warps that are alone already.  The fixed-workspace render,
    whose teams never part, gives the same bits."""
    W, H = 1024, 512
    rng = np.random.default_rng(3)
    counts = rng.integers(33, 65, 2048)
    counts[rng.choice(2048, 10, replace=False)] = 3000
    px, py = _tiles(W, H, 16, counts, 0.3, rng)
    sc = _scene(W, H, px, py, rng.uniform(0.8, 1.5, px.size), 4)
    cam = P.front(W, H)
    p = render.RenderParams(accum=True, stable=True)
    short = np.unique(sc.debug_bins(cam, p)[0], return_counts=True)
    assert short[1][(short[0] > 32) & (short[0] <= 64)].sum() > 2000
    want = sc.render(cam, p)
    for _ in range(20):
        assert torch.equal(sc.render(cam, p), want)
        assert torch.equal(sc.render_noalloc(cam, torch.empty_like(want), p), want)


@pytest.mark.parametrize("T,W,H", [(24, 490, 480), (32, 1000, 520), (40, 1010, 1000)])
def test_regions_off_the_image_do_not_part_teams(T, W, H):
    """Tiles above 16 pixels are rendered as regions of up to 16; those of the last column and row
    can lie wholly off a ragged image.  Every tile's list is long, so every other region is a
    team's, in any order."""
    rng = np.random.default_rng(T)
    nt = -(-W // T) * -(-H // T)
    assert -(-W // T) * T - W >= -(-T // -(-T // 16))  # a column of regions has no pixel
    px, py = _tiles(W, H, T, rng.integers(500, 900, nt), 0.05, rng)
    sc = _scene(W, H, px, py, rng.uniform(0.8, 3.0, px.size), 5)
    cam = P.front(W, H)
    p = render.RenderParams(tile=T, accum=True, stable=True)
    want = sc.render(cam, p)
    for _ in range(20):
        assert torch.equal(sc.render(cam, p), want)
