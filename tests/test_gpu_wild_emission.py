"""Emissions that leave the FP32 range (brightness, colours and view scales are finite each, their
product need not be): the pixels such a particle covers are infinite, all others as without it
(needs a GB300)."""
import numpy as np
import pytest
import torch

import oracle_pins as P
from paper_1606_04427_gb300 import build, render

pytestmark = pytest.mark.gpu

W, H = 70, 45
GREY = np.array([[0.5, 0.4, 0.3], [1.0, 1.0, 1.0]], np.float32)


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    assert torch.cuda.is_available()


def _set(crowd, bright, factor):
    """`crowd` ordinary particles, then `bright` of a species with colours of `factor`."""
    rng = np.random.default_rng(crowd + bright)
    n = crowd + bright
    s = 2.0 / P.focal(H)
    px, py = rng.uniform(0.0, W, n), rng.uniform(0.0, H, n)
    px[crowd:], py[crowd:] = rng.uniform(18.0, 30.0, bright), rng.uniform(2.0, 14.0, bright)
    R = rng.uniform(1.0, 6.0, n)
    R[crowd:] = 3.0
    I = np.where(np.arange(n) < crowd, rng.uniform(0.0, 1.0, n), 0.5)
    return P.make_set(0.5 + (px - 0.5 * W) * s, 0.5 - (py - 0.5 * H) * s, np.full(n, 0.5), R / 0.75 * s, I,
                      type_begin=[0, crowd, n], cmaps=[GREY, GREY * np.float32(factor)], betas=[0.01, 1e30])


def _launch(plan):
    out = plan.new_output()
    plan.launch(out)
    return out.cpu().numpy()


def _check(got, without, covered):
    assert covered.any() and not covered.all()
    assert (got[covered] > 1e18).all()  # a tile split over items holds its sums below 2^62
    np.testing.assert_allclose(got[~covered], without[~covered], rtol=2000 * 2.0 ** -24, atol=1e-12)


# by record counts: alone in short lists, in batches, in a tile split over items
@pytest.mark.parametrize("crowd,bright", [(0, 1), (40, 2), (1500, 3), (60000, 2)])
@pytest.mark.parametrize("kind", ["scene", "vector", "plan", "vector plan"])
def test_infinite_emission_stays_on_covered_pixels(kind, crowd, bright):
    cam = P.front(W, H)
    # where the bright ones cover: their accumulation with ordinary colours
    only = _set(0, bright, 1.0)
    full = _set(crowd, bright, 1e10)
    for name in ("x", "y", "z", "h", "intensity"):
        setattr(only, name, getattr(full, name)[crowd:].copy())
    covered = render.Scene(only, "f32").render(cam, render.RenderParams(accum=True)).cpu().numpy() > 0
    base = _set(crowd, bright, 1e10)
    for name in ("x", "y", "z", "h", "intensity"):
        setattr(base, name, getattr(full, name)[:crowd].copy())
    base.type_begin = np.array([0, crowd, crowd], np.int64)
    if "vector" in kind:  # the ordinary species coloured by a field
        rgb = np.random.default_rng(1).uniform(0.0, 1.0, (crowd + bright, 3)).astype(np.float32)
        for ps in (full, base):
            ps.rgb, ps.col_vector = rgb[:ps.x.shape[0]], np.array([1, 0], np.int32)
    for T in (16, 40):
        p = render.RenderParams(tile=T, accum=True)
        without = render.Scene(base, "f32").render(cam, p).cpu().numpy()
        sc = render.Scene(full, "f32")
        if "plan" in kind:
            got = _launch(render.Plan(sc, [cam], p))[0]
        else:
            got = sc.render(cam, p).cpu().numpy()
        _check(got, without, covered)


def test_a_view_scale_that_overflows():
    """Finite emissions in the scene; the scale of one view makes them infinite there only."""
    cam = P.front(W, H)
    ps = _set(1500, 3, 1.0)
    plan = render.Plan(render.Scene(ps, "f32"), [cam, cam], render.RenderParams(accum=True))
    plan.set_brightness(np.array([[1.0, 1.0], [1.0, 1e20]], np.float32))
    one, two = _launch(plan)
    covered = one > 1e20
    assert np.isfinite(one).all()
    _check(two, one, covered)
