"""Renders of very many small views in one call (needs a GB300): the grids over views and over groups
of views are cut at 65535."""
import dataclasses

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
