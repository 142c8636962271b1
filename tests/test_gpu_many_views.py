"""Renders of very many small views in one call (needs a GB300): the grids over views and over groups
of views are cut at 65535."""
import dataclasses

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


@pytest.mark.parametrize("stable", [False, True])
def test_views_beyond_the_grids_second_dimension(stable):
    ps, cam = P.tiny_scene(5, 24, 8, 8)
    sc = render.Scene(ps, "f32")
    V = 4 * 65535 + 6  # four views per CTA: six views are left for a second launch
    other = [0, 1, 65534, 65535, 65536, V // 2, V - 7, V - 6, V - 5, V - 1]
    cams = [cam] * V
    for k, v in enumerate(other):
        cams[v] = dataclasses.replace(cam, eye=(0.5 + 0.05 * k, 0.45, 2.3 + 0.1 * k))
    p = render.RenderParams(accum=True, stable=stable)
    got = sc.render(cams, p)
    for v in other + [2, 65537, V - 2, V - 3]:
        torch.testing.assert_close(got[v], sc.render(cams[v], p), rtol=24 * 2.0 ** -23, atol=1e-12)


def test_scan_of_more_tiles_than_its_ctas_take_at_once():
    """650 k tiles: every CTA of the scan takes several parts of 4096 tiles one after another; a
    tile of each view is split over items."""
    rng = np.random.default_rng(9)
    W, H, crowd, n = 32, 24, 3000, 3040
    s = 2.0 / P.focal(H)
    px, py = rng.uniform(0.0, W, n), rng.uniform(0.0, H, n)
    px[:crowd], py[:crowd] = 10.5, 9.5
    R = np.where(np.arange(n) < crowd, 0.8, rng.uniform(0.8, 12.0, n))
    sc = render.Scene(P.make_set(0.5 + (px - 0.5 * W) * s, 0.5 - (py - 0.5 * H) * s, np.full(n, 0.5), R / 0.75 * s,
                                 rng.uniform(0.0, 1.0, n), beta=0.001), "f32")
    cam = P.front(W, H)
    V = 850
    other = [0, 3, 424, 848, 849]
    cams = [cam] * V
    for k, v in enumerate(other):
        cams[v] = dataclasses.replace(cam, eye=(0.5 + 0.05 * k, 0.45, 2.3 + 0.1 * k))
    p = render.RenderParams(tile=1, accum=True, timing=True)
    got = sc.render(cams, p)
    assert render.last_timing()["splits"] >= V - len(other)
    for v in other + [1, 2, 500, 847]:
        torch.testing.assert_close(got[v], sc.render(cams[v], p), rtol=n * 2.0 ** -23, atol=1e-12)
