"""Rounding and range of the depth-ordered transfer where a pixel has one record (needs a GB300).
The additive splat evaluates the same weights, so its accumulation is the record's e = E w to the
bit, and I = (1 - exp(-s e)) / s and alpha = exp(-s e) follow in 64 bits."""
import numpy as np
import pytest
import torch

import oracle_pins as P
from paper_1606_04427_gb300 import build, render

pytestmark = pytest.mark.gpu

W = H = 512
CMAP = np.array([[1.0, 0.6, 0.3], [0.0, 0.0, 0.0]], np.float32)


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    assert torch.cuda.is_available()


def _apart(beta):
    """A particle of 5 pixels' support in every 16-pixel tile, all of the first colour (interpolating
    colours rounds in an order that the compiler picks for each kernel), and what it adds."""
    rng = np.random.default_rng(8)
    n = (W // 16) * (H // 16)
    s = 2.0 / P.focal(H)
    px, py = (16.0 * k + rng.uniform(6.0, 10.0, n) for k in divmod(np.arange(n), W // 16))
    ps = P.make_set(0.5 + (px - 0.5 * W) * s, 0.5 - (py - 0.5 * H) * s, np.full(n, 0.5), np.full(n, 5.0 / 0.75 * s),
                    np.zeros(n), cmap=CMAP, beta=beta)
    sc = render.Scene(ps, "f32")
    cam = P.front(W, H)
    return sc, cam, sc.render(cam, render.RenderParams(accum=True)).cpu().numpy()


# beta rounds twice (phi to within 2^-25 of a value above 0.88, the product by 2^-24); before that,
# x's own rounding moves phi by at most x / 2 x 2^-24 = 7.4e-9, the rounding of phi's inner terms by
# 4e-9, and the polynomial is off by 8e-9: 1.2e-7 in all.  Roundings have no sign: over 240000
# values their mean is below 1e-9, and a polynomial's mean error is below its largest.
# For x up to 1, phi is above 0.63 and the inner terms count more: 6.0e-8 for the product, 4.8e-8
# for phi, 3.6e-8 for its inner terms, 2.5e-8 for x's rounding, 9.3e-9 for the polynomial.
@pytest.mark.parametrize("s", [0.3, 1.5, 7.0])
@pytest.mark.parametrize("xmax,tol", [(0.0148, 1.2e-7), (0.04, 1.2e-7), (0.099, 1.2e-7), (0.2, 1.2e-7), (0.249, 1.2e-7),
                                      (0.26, 1.8e-7), (0.99, 1.8e-7)])
def test_one_record_rounds_without_bias(xmax, tol, s):
    sc, cam, e = _apart(xmax / s)
    got = sc.render_ordered(cam, [s]).cpu().numpy().astype(np.float64)
    assert (got[e == 0] == 0).all()
    on = e > 0
    s = float(np.float32(s))
    rel = got[on] * s / -np.expm1(-s * e[on].astype(np.float64)) - 1.0
    assert on.sum() > 200_000
    assert np.abs(rel).max() <= tol
    assert abs(rel.mean()) <= 9e-9


def test_opaque_records_keep_the_precision_of_alpha():
    """alpha = 2^y with y = -s e log2(e) rounded twice beside the constant's rounding: 1.4e-7 y ln 2
    relative for x up to 12, and the exponential's 2^-22."""
    sc, cam, e = _apart(8.0)
    got = sc.render_ordered(cam, [1.5], render.RenderParams(map=True)).cpu().numpy()[..., :3]
    want = np.exp(-1.5 * e.astype(np.float64))
    assert want.min() < 1e-4
    np.testing.assert_allclose(got, want, rtol=1.4e-7 * 12.0 + 2.0 ** -22)


@pytest.mark.parametrize("beta", [1e-30, 1.0, 1e20, 1e30])
def test_species_that_do_not_absorb_at_any_emission(beta):
    sc, cam, e = _apart(beta)
    got = sc.render_ordered(cam, [0.0], render.RenderParams(map=True)).cpu().numpy()
    assert np.array_equal(got[..., 3:], e)
    assert (got[..., :3] == 1.0).all()
