"""Parameters that have run away: what a pixel shows does not depend on the launch
shape that blends it."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_2503_08217_gb300 import scenegen
from paper_2503_08217_gb300.scenegen import make_camera

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2503_08217_gb300 import binding, build
    build.build()
    binding.load()


# four warps per tile, the tile counts at which the lists choose, two warps
@pytest.mark.parametrize("width,height", [(320, 192), (960, 544), (1920, 1088)])
def test_a_splat_without_a_conic_spoils_only_the_pixels_that_reach_it(width, height):
    """A Gaussian whose 2D covariance overflows (along x alone, so that its conic has
    a NaN entry) behind a wall over the left half: pixels that stop at the wall are
    those of the scene without it, the others are NaN. Which stop is read from the
    same scene with a faint plain splat in its place, the last of every list."""
    import gpu_helpers
    wall, count = 24, 25
    g = scenegen.generate("fd", seed=8, n_static=count, n_inst=0, n_steps=2)
    rng = np.random.default_rng(73)
    g.means[:wall] = np.stack([rng.uniform(-4, -3, wall), rng.uniform(-1, 1, wall), np.linspace(4, 6, wall)], 1)
    g.log_scales[:wall] = np.log(2.5)
    g.opacity_logits[:wall] = 3.0                           # 0.953: below the cap of 0.99
    g.means[wall] = (0.3, 0.1, 30.0)
    g.quats[wall] = (1, 0, 0, 0)
    cams = [make_camera(width, height, 0.5 * width, (0.0, 0.0, 0.0), 0.0)]
    g = scenegen.with_cameras(g, [cams, cams])
    vis = oracle.vis_reset(count)[0]

    def run(scales, logit):
        g.log_scales[wall], g.opacity_logits[wall] = scales, logit
        r = gpu_helpers.Renderer(count, 0, cams, max_duplicates=1 << 19)
        return gpu_helpers.gpu_step(g, 0, cams, vis, renderer=r)

    plain, bad, gone = run((5, 5, 5), -5.0), run((45, -3, -3), 0.0), run((-9, -9, -9), -9.0)
    gx = (width + 15) // 16
    tile = (np.arange(height)[:, None] // 16) * gx + np.arange(width)[None] // 16
    length = plain["ranges"][:, 1] - plain["ranges"][:, 0]
    reached = plain["n_contrib"].reshape(height, width) == length[tile]
    assert 0.2 < reached.mean() < 0.9
    image = bad["images"][0]
    # a pixel within a hundredth of its stop may go either way
    sure = ~((gone["final_T"].reshape(height, width) >= 1e-4) & (gone["final_T"].reshape(height, width) < 1.01e-4))
    assert np.isnan(image[:, reached & sure]).all()
    np.testing.assert_array_equal(image[:, ~reached & sure], gone["images"][0][:, ~reached & sure])
