"""The splat's batches and passes at the sizes where they change (needs a GB300): one warp
renders a region of up to 16 x 16 pixels from batches of 192 records, read 32 at a time,
and evaluates 16 squares of 4 x 4 pixels per pass."""
import numpy as np
import pytest
import torch

import oracle
import oracle_pins as P
from paper_1606_04427_gb300 import build, render

pytestmark = pytest.mark.gpu

W, H = 40, 27  # the last regions are partial in both directions for every tile below


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    assert torch.cuda.is_available()


def _at(px, py):
    """World x, y of image position (px, py) on the plane z = 0.5 (camera depth 2)."""
    s = 2.0 / P.focal(H)
    return 0.5 + (np.asarray(px) - 0.5 * W) * s, 0.5 - (np.asarray(py) - 0.5 * H) * s


def _layout(kind, n, rng):
    """(image x, image y, support radius in pixels)."""
    if kind == "pixel":        # every record in one square: its pairs of lanes share the list
        return np.full(n, 18.3), np.full(n, 9.6), np.full(n, 0.8)
    if kind == "square":
        return rng.uniform(20.0, 24.0, n), rng.uniform(8.0, 12.0, n), rng.uniform(0.8, 2.0, n)
    if kind == "spread":
        return rng.uniform(-3.0, W + 3.0, n), rng.uniform(-3.0, H + 3.0, n), rng.uniform(0.75, 9.0, n)
    return rng.uniform(0.0, W, n), rng.uniform(0.0, H, n), rng.uniform(20.0, 60.0, n)


def _set(kind, n, seed):
    rng = np.random.default_rng(seed)
    px, py, R = _layout(kind, n, rng)
    x, y = _at(px, py)
    return P.make_set(x, y, np.full(n, 0.5), R / 0.75 * 2.0 / P.focal(H), rng.uniform(0.0, 1.0, n), beta=0.01)


# A pixel sums at most n non-negative terms in FP32, within (n - 1) 2^-24 of the exact sum
# whatever the order.  A term's weight is 2^a with a in [-5.8, 0]: a's roundings (distance,
# scale, product; about five of 2^-24) move it by 5.8 x 5 x 2^-24 x ln 2 = 1.2e-6, the
# exponential by 2^-22, the colour code (24 bits) by less than 1e-6.
def _rtol(n):
    return (n - 1) * 2.0 ** -24 + 4e-6


@pytest.mark.parametrize("kind", ["pixel", "square", "spread", "large"])
@pytest.mark.parametrize("n", [1, 32, 33, 97, 191, 192, 193, 385])
def test_batch_edges_match_the_oracle(kind, n):
    ps = _set(kind, n, n)
    cam = P.front(W, H)
    want = oracle.render(ps, cam)
    sc = render.Scene(ps, "f32")
    for T in (5, 16, 24, 33, 64):
        got = sc.render(cam, render.RenderParams(tile=T, accum=True)).cpu().numpy()
        np.testing.assert_allclose(got, want, rtol=_rtol(n), atol=1e-12, err_msg=f"{kind} n={n} T={T}")


def test_supports_whose_square_leaves_the_fp32_range():
    """Radii whose square underflows cover nothing or their own pixel centre, radii whose
    square overflows cover every pixel with weight one: never a NaN."""
    n = 6
    px, py = np.array([3.5, 10.2, 20.5, 30.5, 8.0, 25.0]), np.array([4.5, 12.0, 20.5, 5.5, 3.0, 15.0])
    x, y = _at(px, py)
    h = np.array([1e-25, 1e-30, 0.01, 1e-22, 1e18, 1e19])
    ps = P.make_set(x, y, np.full(n, 0.5), h, np.full(n, 0.5), beta=0.1)
    cam = P.front(W, H)
    got = render.Scene(ps, "f32").render(cam, render.RenderParams(r_min_px=0.0, accum=True)).cpu().numpy()
    assert np.isfinite(got).all()
    want = oracle.render(ps, cam, oracle.Params(r_min_px=0.0))
    np.testing.assert_allclose(got, want, rtol=_rtol(n), atol=1e-12)


@pytest.mark.parametrize("emax", [0.03, 0.06, 0.19, 0.24, 3.0])
@pytest.mark.parametrize("kind,n", [("pixel", 193), ("square", 97), ("spread", 385), ("large", 64), ("large", 1)])
def test_ordered_batch_edges_match_the_oracle(kind, n, emax):
    """Batches of the depth-ordered splat, on every polynomial degree of the transfer and at
    its limits (x up to 0.04, 0.2 and beyond), beside a species that does not absorb."""
    rng = np.random.default_rng(n)
    px, py, R = _layout(kind, n, rng)
    x, y = _at(px, py)
    half = n // 2
    ps = P.make_set(x, y, rng.permutation(np.linspace(0.49, 0.51, n)), R / 0.75 * 2.0 / P.focal(H),
                    rng.uniform(0.0, 1.0, n), type_begin=[0, half, n], betas=[emax, emax])
    cam = P.front(W, H)
    sc = render.Scene(ps, "f32")
    absorb = [1.0, 0.0]
    want = oracle.render_rt_depth(ps, cam, absorb)
    # the weights' relative error 2.5e-6 (above) reaches I through each emission and through
    # the absorption in front of it, at most tau of it; each of n updates rounds three times
    # and its u is off by 1.2e-7 at most
    tau = oracle.render(ps, cam).max()
    rtol = 4e-6 * (1.0 + tau) + n * (3 * 2.0 ** -24 + 1.2e-7)
    for T in (5, 16, 24, 32):
        got = sc.render_ordered(cam, absorb, render.RenderParams(tile=T)).cpu().numpy()
        np.testing.assert_allclose(got, want, rtol=rtol, atol=1e-12, err_msg=f"{kind} n={n} T={T}")
