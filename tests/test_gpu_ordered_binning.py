"""The depth-ordered binning at its edges (needs a GB300): one particle, no active one, keys that
span nothing, one byte or all bits, particles of one to several tiles."""
import numpy as np
import pytest
import torch

import oracle
import oracle_pins as P
from paper_1606_04427_gb300 import build, render

pytestmark = pytest.mark.gpu

W, H = 200, 90


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()
    assert torch.cuda.is_available()


# As for the ordered splat's batches: the weights' relative error 2.5e-6 reaches a pixel through
# each emission and the absorption in front of it (at most tau of it); each of n updates rounds
# three times and its u is off by 1.2e-7 at most.
@pytest.mark.parametrize("depth", ["equal", "near", "wide", "behind"])
@pytest.mark.parametrize("n", [1, 2, 33, 4097])
def test_ordered_binning_edges_match_the_oracle(n, depth):
    rng = np.random.default_rng(n)
    z = {"equal": np.full(n, 0.5), "near": rng.uniform(0.4999, 0.5001, n),
         "wide": 2.5 - 2.0 ** rng.uniform(-9.0, 6.0, n), "behind": np.full(n, 3.0)}[depth]
    if depth == "behind" and n > 2:
        z[n // 2] = 0.5  # one active particle
    s = (2.5 - z) / P.focal(H)  # world units per pixel at depth 2.5 - z
    px, py = rng.uniform(0.0, W, n), rng.uniform(0.0, H, n)
    R = np.where(rng.random(n) < 0.9, rng.uniform(0.8, 4.0, n), rng.uniform(8.0, 60.0, n))
    ps = P.make_set(0.5 + (px - 0.5 * W) * s, 0.5 - (py - 0.5 * H) * s, z, np.abs(R / 0.75 * s),
                    rng.uniform(0.0, 1.0, n), beta=0.02)
    cam = P.front(W, H)
    want = oracle.render_rt_depth(ps, cam, [1.0])
    rtol = 4e-6 * (1.0 + oracle.render(ps, cam).max()) + n * (3 * 2.0 ** -24 + 1.2e-7)
    sc = render.Scene(ps, "f32")
    for T in (8, 16, 32):
        got = sc.render_ordered(cam, [1.0], render.RenderParams(tile=T)).cpu().numpy()
        np.testing.assert_allclose(got, want, rtol=rtol, atol=1e-12, err_msg=f"T={T}")


@pytest.mark.parametrize("n", [513, 8192, 9001])  # 2, 16 and 18 slices of the tile at (16, 16)
@pytest.mark.parametrize("T", [16, 20, 24, 32])
def test_slices_of_a_crowded_tile_compose_far_to_near(n, T):
    rng = np.random.default_rng(n)
    z = rng.uniform(0.49, 0.51, n)
    s = (2.5 - z) / P.focal(H)
    px, py, R = rng.uniform(18.0, 30.0, n), rng.uniform(18.0, 30.0, n), rng.uniform(0.8, 5.0, n)
    ps = P.make_set(0.5 + (px - 0.5 * W) * s, 0.5 - (py - 0.5 * H) * s, z, R / 0.75 * s,
                    rng.uniform(0.0, 1.0, n), beta=0.01)
    cam = P.front(W, H)
    want = oracle.render_rt_depth(ps, cam, [1.0])
    rtol = 4e-6 * (1.0 + oracle.render(ps, cam).max()) + n * (3 * 2.0 ** -24 + 1.2e-7)
    sc = render.Scene(ps, "f32")
    got = sc.render_ordered(cam, [1.0], render.RenderParams(tile=T)).cpu().numpy()
    np.testing.assert_allclose(got, want, rtol=rtol, atol=1e-12)
    maps = sc.render_ordered(cam, [1.0], render.RenderParams(tile=T, map=True)).cpu().numpy()
    np.testing.assert_array_equal(maps[..., 3:], got)
    # with absorption equal to emission, I = 1 - alpha
    np.testing.assert_allclose(1.0 - maps[..., :3], want, rtol=rtol, atol=n * 2.0 ** -23)
