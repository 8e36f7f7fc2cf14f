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


@pytest.mark.parametrize("count,extent", [(300_000, 0.95), (20_000, 0.02)], ids=["even", "long_list"])
def test_forward_queue_forms_agree(count, extent):
    """One image as 1, 2 and 3 copies: four warps per tile and a CTA for every tile;
    the tile counts at which the lists choose between two and four warps (evenly
    filled tiles, or nearly all splats in a few tiles); two warps and tiles drawn
    from the cursor. With the even lists there are more clearing chunks (2,048
    splats) than CTAs without a tile. Same pixels and last contributors, gradients
    in proportion, also in a second step (cursor and splat adjoints are back at zero)."""
    import gpu_helpers
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(67)
    g = scenegen.generate("fd", seed=6, n_static=count, n_inst=0, n_steps=2)
    z = rng.uniform(4, 12, count)
    g.means[:] = np.stack([rng.uniform(-extent, extent, count) * z, rng.uniform(-0.8 * extent, 0.8 * extent, count) * z, z], 1)
    g.log_scales[:] = np.log(rng.uniform(0.002, 0.02, (count, 3)))
    rows = 9 * sms // 40                                    # 40 x rows tiles, at most 9 CTAs per SM
    cam = make_camera(640, 16 * rows, 320.0, (0.0, 0.0, 0.0), 0.0)
    g = scenegen.with_cameras(g, [[cam], [cam]])
    vis = oracle.vis_reset(count)[0]
    d = rng.standard_normal((3, cam.height, cam.width))
    P = cam.width * cam.height
    first = None
    for copies in (1, 2, 3):
        cams = [cam] * copies
        r = gpu_helpers.Renderer(g.n, 0, cams, max_splats=count * copies, max_duplicates=16 * count)
        for _ in range(2):
            res = gpu_helpers.gpu_step(g, 0, cams, vis, dL=[d / copies] * copies, renderer=r)
            chunks, tiles, pairs = -(-res["counts"]["n_splats"] // 2048), 40 * rows * copies, res["counts"]["n_duplicates"]
            assert (copies > 1) == (tiles > 9 * sms) and (copies > 2) == (tiles > 18 * sms)
            longest = int((res["ranges"][:, 1] - res["ranges"][:, 0]).max())
            if extent > 0.5:
                assert chunks > 9 * sms - 40 * rows and pairs > 300_000
            else:
                assert pairs < 300_000 and longest * tiles > 6 * pairs
            first = first or res
            for v in range(copies):
                np.testing.assert_allclose(res["images"][v], first["images"][0], rtol=0, atol=1e-6)
                np.testing.assert_array_equal(res["n_contrib"][v * P:(v + 1) * P], first["n_contrib"][:P])
            for k, a in first["grads"].items():
                if a.size:
                    np.testing.assert_allclose(res["grads"][k], a, rtol=1e-4, atol=5e-5 * max(np.abs(a).max(), 1e-30),
                                               err_msg=k)


@pytest.mark.parametrize("values", [1, 4, 1000])
def test_sort_of_coarse_depths(values):
    """Depths of few values, their low digits multiples of 64 (a flat wall, and a
    scene far from the origin): equal depths keep the splats' order."""
    import gpu_helpers
    from test_gpu_parity import _stage_isolated_sort
    count = 9000
    rng = np.random.default_rng(values)
    g = scenegen.generate("fd", seed=7, n_static=count, n_inst=0, n_steps=2)
    z = (16.0 + rng.integers(0, values, count) * 2.0 ** -13).astype(np.float32)
    g.means[:] = np.stack([rng.uniform(-0.9, 0.9, count) * z, rng.uniform(-0.9, 0.9, count) * z, z], 1)
    g.log_scales[:] = np.log(0.05)
    cams = [make_camera(480, 480, 240.0, (0.0, 0.0, 0.0), 0.0)]
    g = scenegen.with_cameras(g, [cams, cams])
    res = gpu_helpers.gpu_step(g, 0, cams, oracle.vis_reset(count)[0])
    assert res["counts"]["n_splats"] > count // 2
    depth = np.unique(res["rgb_d"][:, 3].view(np.uint32))
    assert depth.size <= values and not (depth & 63).any()
    _stage_isolated_sort(res, cams)


def test_pose_adjoint_of_a_large_instance_keeps_its_precision():
    """One instance of 400,000 Gaussians beside 259 empty ones (1,566 matrices, near
    the most a call takes): its pose adjoint against the FP64 sum of those of the
    same Gaussians as 100 instances with the same pose. Partial sums per CTA gave a
    mean error of 5.2e-7 of the largest entry, 20 partial sums 1.3e-6; the bound is
    one and a half times the former."""
    from paper_2503_08217_gb300.render import DeviceScene, Renderer
    static, count, parts = 2000, 400_000, 100
    gen = torch.Generator(device="cuda")
    gen.manual_seed(71)
    n = static + count
    uni = lambda lo, hi, *s: torch.empty(s, device="cuda").uniform_(lo, hi, generator=gen)        # noqa: E731
    means = torch.stack([uni(-20, 20, n), uni(-2, 15, n), uni(0, 60, n)], 1)
    means[static:] = torch.stack([uni(-8, 8, count), uni(-3, 3, count), uni(-8, 8, count)], 1)
    quats = torch.empty(n, 4, device="cuda").normal_(generator=gen)
    scene = DeviceScene(means=means.contiguous(), log_scales=torch.full((n, 3), -3.5, device="cuda"),
                        quats=(quats / quats.norm(dim=1, keepdim=True)).contiguous(),
                        opacity_logits=torch.empty(n, device="cuda").normal_(generator=gen),
                        sh=torch.empty(n, 4, 3, device="cuda").normal_(0, 0.3, generator=gen),
                        inst_offsets=torch.zeros(3, dtype=torch.int64, device="cuda"), sh_degree=1)
    cams = [make_camera(640, 360, 320.0, (0.0, 0.0, 30.0), 2 * np.pi * k / 6) for k in range(6)]
    pixels = 6 * 640 * 360
    dL = torch.empty(3 * pixels, device="cuda").normal_(0, 1.0 / pixels, generator=gen)
    window = torch.tensor([-1.0, 1.0], device="cuda").repeat(n, 1).contiguous()
    bg = torch.zeros(3, device="cuda")

    def adjoint(offsets, n_inst):
        scene.inst_offsets = torch.tensor(offsets, dtype=torch.int64, device="cuda")
        quat = torch.tensor([[0.999, 0.0, 0.0447, 0.0]], device="cuda").repeat(n_inst, 1).contiguous()
        trans = torch.tensor([[0.3, 1.0, 30.2]], device="cuda").repeat(n_inst, 1).contiguous()
        r = Renderer(n, n_inst, cams, max_splats=6 * n, max_duplicates=1 << 24)
        r.forward(scene, quat, trans, cams, 0.0, window, None, 0.5, bg)
        grads = {k: torch.zeros_like(t) for k, t in zip(("means", "log_scales", "quats", "opacity_logits", "sh",
                                                         "inst_quat", "inst_trans"), scene.params() + [quat, trans])}
        r.backward(scene, quat, trans, bg, dL, grads)
        r.sync_status()
        g = torch.cat([grads["inst_quat"], grads["inst_trans"]], 1).double().cpu().numpy()
        assert r.counts()["n_splats"] > count // 2
        return g

    split = [0] + [static + k * (count // parts) for k in range(parts)] + [n]
    want = np.mean([adjoint(split, parts).sum(0) for _ in range(3)], 0)
    errors = []
    for _ in range(6):
        g = adjoint([0, static] + [n] * 260, 260)
        assert not g[1:].any()
        errors.append(np.abs(g[0] - want).max() / np.abs(want).max())
    assert np.mean(errors) <= 8e-7, errors


@pytest.mark.parametrize("n_inst", [1, 3, 4, 5, 4001])
def test_world_adjoints_of_tiny_instances(n_inst):
    """Instances of 0 to 2 Gaussians, whole and broken groups of the four that a CTA
    maps to poses: dt is the sum of the rows' adjoints, equal poses with equal rows
    get equal adjoints, empty instances zero, and a second call repeats the first
    (the sums were cleared)."""
    from paper_2503_08217_gb300 import binding
    from paper_2503_08217_gb300.render import Renderer
    rng = np.random.default_rng(n_inst)
    sizes = np.arange(n_inst) % 3
    off = np.r_[0, 7, 7 + np.cumsum(sizes)].astype(np.int64)
    n = int(off[-1])
    cu = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()   # noqa: E731
    f32 = lambda *s: rng.standard_normal(s).astype(np.float32)        # noqa: E731
    means, quats, sh = cu(f32(n, 3)), cu(f32(n, 4)), cu(f32(n, 16, 3))
    pq, pt = cu(np.tile(f32(1, 4), (n_inst, 1))), cu(f32(n_inst, 3))
    log_scales, logits, offsets = cu(f32(n, 3)), cu(f32(n)), cu(off)      # held: the scene keeps addresses only
    cs = binding.make_scene(means, log_scales, quats, logits, sh, offsets, 3)
    poses = binding.make_poses(pq, pt)
    r = Renderer(n, n_inst, [make_camera(16, 16, 14.0, (0.0, 0.0, 0.0), 0.0)])
    up = {"means": f32(n, 3), "quats": f32(n, 4), "sh": f32(n, 16, 3)}
    got = []
    for _ in range(2):
        g = {k: cu(v) for k, v in up.items()}
        g["inst_quat"] = torch.full((n_inst, 4), float("nan"), device="cuda")
        g["inst_trans"] = torch.full((n_inst, 3), float("nan"), device="cuda")
        r.ws.to_world_bwd(cs, poses, g)
        got.append({k: v.cpu().numpy() for k, v in g.items()})
    want = np.array([up["means"][off[k + 1]:off[k + 2]].sum(0) for k in range(n_inst)])
    np.testing.assert_allclose(got[0]["inst_trans"], want, rtol=0, atol=1e-6)
    assert not got[0]["inst_quat"][sizes == 0].any()
    if (sizes > 0).any():
        assert np.abs(got[0]["inst_quat"][sizes > 0]).max(axis=1).min() > 0
    for k in got[0]:
        np.testing.assert_array_equal(got[0][k], got[1][k])


@pytest.mark.parametrize("K,D,S", [(1, 1, 1), (3, 16, 2), (70, 8, 1)])
def test_ode_trajectory_without_steps(K, D, S):
    """One output time: the poses are the initial states' own, only they get a
    gradient, and every other gradient stays exactly what it was."""
    from paper_2503_08217_gb300 import binding
    from oracle import ode
    cu = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()   # noqa: E731
    params, embed, z0 = scenegen.ode_model(79, K, D)
    rng = np.random.default_rng(83)
    times = np.array([0.3], np.float32)
    p, e, z, t = cu(params), cu(embed), cu(z0), cu(times)
    states, quat, trans = binding.ode_poses(p, e, z, t, S)
    np.testing.assert_array_equal(states.cpu().numpy().reshape(-1), z0.reshape(-1))
    np.testing.assert_array_equal(trans.cpu().numpy().reshape(K, 3), z0[:, :3])
    gq, gt = rng.standard_normal((1, K, 4)).astype(np.float32), rng.standard_normal((1, K, 3)).astype(np.float32)
    g_params, g_embed = torch.full((params.size,), 0.5, device="cuda"), torch.full((K, D), -0.25, device="cuda")
    g_z0 = torch.zeros((K, 6), device="cuda")
    gq_t, gt_t = cu(gq), cu(gt)
    binding.ode_poses_bwd(p, e, t, S, states, gq_t, gt_t, g_params, g_embed, g_z0)
    torch.cuda.synchronize()
    assert (g_params == 0.5).all() and (g_embed == -0.25).all()
    want = ode.backward(params, embed, z0, times, S, 64, gq.astype(np.float64), gt.astype(np.float64))[2]
    a = g_z0.double().cpu().numpy()
    np.testing.assert_array_equal(a[:, :3], gt[0])
    assert np.linalg.norm(a - want) <= 1e-5 * np.linalg.norm(want)


def test_captured_forward_chooses_at_replay():
    """A forward captured on evenly filled tiles and replayed on splats massed in a
    few (and back) renders what a call does: which launch works is decided on the
    device. The images have tile counts at which the lists choose."""
    import gpu_helpers
    from paper_2503_08217_gb300.render import DeviceScene
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rows = 14 * sms // 40                                   # 40 x rows tiles, between 9 and 18 per SM
    count = 20_000
    rng = np.random.default_rng(89)
    g = scenegen.generate("fd", seed=9, n_static=count, n_inst=0, n_steps=2)
    cam = make_camera(640, 16 * rows, 320.0, (0.0, 0.0, 0.0), 0.0)
    g = scenegen.with_cameras(g, [[cam], [cam]])
    g.log_scales[:] = np.log(rng.uniform(0.005, 0.03, (count, 3)))
    z = rng.uniform(4, 12, count)
    xy = rng.uniform(-1, 1, (count, 2)) * z[:, None]
    places = [np.concatenate([e * xy, z[:, None]], 1).astype(np.float32) for e in (0.95, 0.02)]
    g.means[:] = places[0]
    dev = DeviceScene.from_host(g)
    vis = torch.from_numpy(oracle.vis_reset(count)[0]).cuda()
    bg = torch.tensor([0.2, 0.4, 0.6], device="cuda")
    iq = torch.from_numpy(np.ascontiguousarray(g.inst_quat[0], np.float32)).cuda()
    it = torch.from_numpy(np.ascontiguousarray(g.inst_trans[0], np.float32)).cuda()
    make = lambda: gpu_helpers.Renderer(count, 0, [cam], max_duplicates=1 << 20)      # noqa: E731
    r, eager = make(), make()
    out = torch.empty(3 * cam.width * cam.height, device="cuda")
    graph = r.capture(lambda: r.forward(dev, iq, it, [cam], 0.0, vis, None, 0.0, bg, out))
    for place in (0, 1, 0, 1):
        dev.means.copy_(torch.from_numpy(places[place]).cuda())
        out.fill_(float("nan"))
        graph.replay()
        want = eager.forward(dev, iq, it, [cam], 0.0, vis, None, 0.0, bg)
        torch.cuda.synchronize()
        ranges = r.ws.debug("tile_ranges", torch.int32, 80 * rows).view(-1, 2)
        longest, pairs = int((ranges[:, 1] - ranges[:, 0]).max()), r.counts()["n_duplicates"]
        assert (longest * 40 * rows > 6 * pairs) == (place == 1) and pairs < 300_000
        np.testing.assert_array_equal(out.cpu().numpy(), want.cpu().numpy())
