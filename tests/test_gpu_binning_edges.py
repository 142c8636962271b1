"""Tile lists at the sizes where the binning changes (needs a GB300): rounds of 1024 particles,
windows of 4096 staged pairs, one or two sort passes (up to 128 tiles per view, or more),
candidate boxes of 2 x 2 tiles, within a block of 8 x 4 and beyond it."""
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


@pytest.mark.parametrize("size,tile", [((64, 40), 8), ((176, 176), 16), ((177, 176), 16), ((640, 512), 5)])
@pytest.mark.parametrize("n,radius", [(1, 3.0), (1023, 6.0), (1024, 6.0), (1025, 6.0), (2500, 30.0)])
@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_lists_match_the_oracle(size, tile, n, radius, storage):
    W, H = size
    rng = np.random.default_rng(n + W)
    scale = 2.0 / P.focal(H)  # world units per pixel on the plane z = 0.5
    x = 0.5 + (rng.uniform(-20.0, W + 20.0, n) - 0.5 * W) * scale
    y = 0.5 + (rng.uniform(-20.0, H + 20.0, n) - 0.5 * H) * scale
    h = rng.uniform(0.3, 1.0, n) ** 3 * radius / 0.75 * scale
    ps = P.make_set(x, y, np.full(n, 0.5), h, rng.uniform(0.0, 1.0, n))
    cam = P.front(W, H)
    counts, offsets, members = render.Scene(ps, storage).debug_bins(cam, render.RenderParams(tile=tile))
    c, o, m = oracle.bins(ps, cam, oracle.Params(tile=tile), storage)
    np.testing.assert_array_equal(counts, c)
    np.testing.assert_array_equal(offsets, o)
    np.testing.assert_array_equal(members, m)
