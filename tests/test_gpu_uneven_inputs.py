"""Inputs whose work is spread unevenly: kernels that share it out by an average
have to stay within bounds, and correct, where one part holds nearly all of it.

Times are compared with those of kernels of the same call that visit every
splat once, with bounds several times above what a pass over the splats takes
and far below what one CTA walking all of them took.
"""
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


def _kernel_times(scene, cams, vis, renderer, repeats=5):
    """Median kernel times (ms) of a forward."""
    import gpu_helpers
    renderer.ws.set_timing(True)
    seen = []
    for _ in range(repeats):
        gpu_helpers.gpu_step(scene, 0, cams, vis, renderer=renderer)
        seen.append(renderer.ws.kernel_times())
    renderer.ws.set_timing(False)
    return {k: float(np.median([s[k] for s in seen])) for k in seen[0]}


def test_faint_splats_behind_the_last_pair():
    """Splats too faint for any tile behind all that have pairs: the last chunk of
    the pair expansion does not walk them (at 400,000 of them one CTA took about
    1 ms, the scan of all counts 0.015 ms)."""
    import gpu_helpers
    from test_gpu_parity import _stage_isolated_sort
    near, count = 300, 400_000
    rng = np.random.default_rng(61)
    g = scenegen.generate("fd", seed=4, n_static=count, n_inst=0, n_steps=2)
    z = np.r_[rng.uniform(4, 8, near), rng.uniform(20, 40, count - near)]
    g.means[:] = np.stack([rng.uniform(-0.9, 0.9, count) * z, rng.uniform(-0.9, 0.9, count) * z, z], 1)
    g.log_scales[:] = np.log(0.02)
    g.opacity_logits[:] = -8.0                              # opacity 3e-4 < 1/255
    g.opacity_logits[:near] = 1.0
    cams = [make_camera(320, 320, 160.0, (0.0, 0.0, 0.0), 0.0)]
    g = scenegen.with_cameras(g, [cams, cams])
    vis = oracle.vis_reset(count)[0]
    r = gpu_helpers.Renderer(g.n, 0, cams, max_duplicates=1 << 20)
    res = gpu_helpers.gpu_step(g, 0, cams, vis, renderer=r)
    assert res["counts"]["n_splats"] > count // 2 and near <= res["counts"]["n_duplicates"] < 20 * near
    _stage_isolated_sort(res, cams)
    ms = _kernel_times(g, cams, vis, r)
    assert ms["duplicate_expand"] <= 10 * ms["duplicate"], ms
