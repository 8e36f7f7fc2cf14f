"""The sizes at which a kernel changes its path or its last block is ragged.

Tolerances, all FP32 against FP64 or against the same path at another size:
  * selections, visibility records, pair lists: equal;
  * images of the same splats by another launch shape: 1e-6 (the same
    operations per pixel; three products of values up to 1 are added per splat);
  * NeuralODE states: 2e-5 (1 + |z|), gradients 1e-3 relative per tensor, as in
    the file on the NeuralODE;
  * world transform: an output is a sum of at most 7 products with matrix
    entries, each a 26-term FP32 sum (26 x 6e-8 = 1.6e-6), so 2e-5 of the
    tensor's largest value; pose sums add at most 95 x 48 such terms in FP32,
    1e-4 relative per tensor;
  * gradients of one scene by two routes: the per-splat sums are float atomics
    in another order, so 1e-4 of the element and 5e-5 of the tensor's largest.
"""
from __future__ import annotations

import copy

import numpy as np
import pytest

import oracle
from oracle import ode
from paper_2503_08217_gb300 import scenegen
from paper_2503_08217_gb300.scenegen import make_camera

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

NAMES = ("means", "log_scales", "quats", "opacity_logits", "sh", "inst_quat", "inst_trans")


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2503_08217_gb300 import binding, build
    build.build()
    binding.load()


def _cu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _rel(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-30))


def _close_grads(a, b):
    for k in NAMES:
        scale = max(np.abs(b[k]).max(), 1e-30)
        np.testing.assert_allclose(a[k], b[k], rtol=1e-4, atol=5e-5 * scale, err_msg=k)


# ------------------------------------------------------------------ NeuralODE
# the backward's pipeline takes two steps a tick: no step, one, an odd number,
# a full tick; one instance; no embedding and the widest
@pytest.mark.parametrize("K,D,S,T", [(1, 0, 1, 1), (2, 16, 1, 2), (1, 3, 3, 2), (3, 16, 2, 3), (1, 0, 1, 6)])
def test_ode_short_trajectories(K, D, S, T):
    from paper_2503_08217_gb300 import binding
    params, embed, z0 = scenegen.ode_model(17, K, D)
    z0[:, 3:] = np.random.default_rng(18).uniform(-0.4, 0.4, (K, 3)).astype(np.float32)
    times = np.linspace(-0.5, 0.7, T).astype(np.float32)
    states, quat, trans = binding.ode_poses(_cu(params), _cu(embed), _cu(z0), _cu(times), S)
    st_o = ode.trajectory(params, embed, z0, times, S, 64)
    q_o, t_o = ode.poses(st_o, S)
    st = states.double().cpu().numpy()
    assert (np.abs(st - st_o) <= 2e-5 * (1.0 + np.abs(st_o))).all()
    np.testing.assert_allclose(quat.double().cpu().numpy(), q_o, rtol=0, atol=2e-5)
    np.testing.assert_allclose(trans.double().cpu().numpy(), t_o, rtol=2e-5, atol=2e-5)
    rng = np.random.default_rng(19)
    gq = rng.standard_normal((T, K, 4)).astype(np.float32)
    gt = rng.standard_normal((T, K, 3)).astype(np.float32)
    g = [torch.zeros(params.size, device="cuda"), torch.zeros((K, D), device="cuda"),
         torch.zeros((K, 6), device="cuda")]
    binding.ode_poses_bwd(_cu(params), _cu(embed), _cu(times), S, states, _cu(gq), _cu(gt), *g)
    torch.cuda.synchronize()
    want = ode.backward(params, embed, z0, times, S, 64, gq.astype(np.float64), gt.astype(np.float64))
    for name, a, b in zip(("params", "embed", "z0"), g, want):
        assert _rel(a.double().cpu().numpy(), b) <= 1e-3 or not b.size or not np.abs(b).max(), name
        if T == 1 and name == "params":
            assert not a.any()


# ------------------------------------------------------------ world transform
def _rotation(q):
    w, x, y, z = np.moveaxis(q / np.linalg.norm(q, axis=-1, keepdims=True), -1, 0)
    return np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                     2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                     2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], -1).reshape(q.shape[:-1] + (3, 3))


def _hamilton(p, q):
    a, b, c, d = np.moveaxis(p, -1, 0)
    e, f, g, h = np.moveaxis(q, -1, 0)
    return np.stack([a * e - b * f - c * g - d * h, a * f + b * e + c * h - d * g,
                     a * g - b * h + c * e + d * f, a * h + b * g - c * f + d * e], -1)


_DIRS = np.random.default_rng(23).standard_normal((64, 3))
_DIRS /= np.linalg.norm(_DIRS, axis=1, keepdims=True)


def _sh_matrix(R, K):
    """D with Y(R^T d) = D Y(d), by least squares over 64 directions."""
    Y = np.stack([oracle.sh_basis(d)[0][:K] for d in _DIRS])
    Yr = np.stack([oracle.sh_basis(R.T @ d)[0][:K] for d in _DIRS])
    return np.linalg.lstsq(Y, Yr, rcond=None)[0].T


def _world(off, means, quats, sh, pq, pt):
    """The dynamic rows of the transform in FP64."""
    m, q, c = means.copy(), quats.copy(), sh.copy()
    for k in range(len(off) - 2):
        s = slice(off[k + 1], off[k + 2])
        R = _rotation(pq[k])
        m[s] = means[s] @ R.T + pt[k]
        q[s] = _hamilton(np.broadcast_to(pq[k] / np.linalg.norm(pq[k]), quats[s].shape),
                         quats[s] / np.linalg.norm(quats[s], axis=1, keepdims=True))
        D = _sh_matrix(R, sh.shape[1])
        c[s] = np.einsum("ji,njc->nic", D, sh[s])
    return m, q, c


# a warp takes 32 rows of one instance at a time
@pytest.mark.parametrize("degree", [0, 1, 2, 3])
def test_world_transform_ragged_instances(degree):
    from paper_2503_08217_gb300 import binding
    sizes = [5, 1, 0, 31, 32, 33, 0, 95, 64]               # static rows first
    off = np.r_[0, np.cumsum(sizes)].astype(np.int64)
    n, n_inst, K = int(off[-1]), len(sizes) - 1, (degree + 1) ** 2
    rng = np.random.default_rng(29 + degree)
    f32 = lambda *s: rng.standard_normal(s).astype(np.float32)   # noqa: E731
    means, quats, sh, pq, pt = f32(n, 3), f32(n, 4), f32(n, K, 3), f32(n_inst, 4), f32(n_inst, 3)
    gm, gq, gs = f32(n, 3), f32(n, 4), f32(n, K, 3)
    one = torch.zeros((n, 3), device="cuda")
    dm, dq, ds, do = _cu(means), _cu(quats), _cu(sh), _cu(off)
    cs = binding.make_scene(dm, one, dq, torch.zeros(n, device="cuda"), ds, do, degree)
    tq, tt = _cu(pq), _cu(pt)
    poses = binding.make_poses(tq, tt)
    out = [dm.clone(), dq.clone(), ds.clone()]
    binding.to_world(cs, poses, *out)
    d64 = [a.astype(np.float64) for a in (means, quats, sh, pq, pt)]
    want = _world(off, *d64)
    for a, b in zip(out, want):
        np.testing.assert_allclose(a.double().cpu().numpy(), b, rtol=0, atol=2e-5 * np.abs(b).max())

    # backward: FP64 differences of the loss sum <g, world rows>, whose error is
    # about 1e-9; means and SH enter linearly
    g64 = [a.astype(np.float64) for a in (gm, gq, gs)]
    rows = lambda w: sum((g * x).reshape(n, -1).sum(1) for g, x in zip(g64, w))   # noqa: E731
    h = 1e-5
    e_q, e_pq, e_pt = np.zeros((n, 4)), np.zeros((n_inst, 4)), np.zeros((n_inst, 3))
    segment = [slice(off[k + 1], off[k + 2]) for k in range(n_inst)]
    for i in range(4):
        d = h * np.eye(4)[i]
        m_, q_, s_, p_, t_ = d64
        e_q[:, i] = (rows(_world(off, m_, q_ + d, s_, p_, t_)) - rows(_world(off, m_, q_ - d, s_, p_, t_))) / (2 * h)
        diff = (rows(_world(off, m_, q_, s_, p_ + d, t_)) - rows(_world(off, m_, q_, s_, p_ - d, t_))) / (2 * h)
        e_pq[:, i] = [diff[s].sum() for s in segment]
    e_m, e_s = g64[0].copy(), g64[2].copy()
    for k, s in enumerate(segment):
        R = _rotation(d64[3][k])
        e_m[s] = g64[0][s] @ R
        e_s[s] = np.einsum("ij,njc->nic", _sh_matrix(R, K), g64[2][s])
        e_pt[k] = g64[0][s].sum(0)
    e_q[:off[1]] = g64[1][:off[1]]                          # static rows are not touched
    cams = [make_camera(16, 16, 14.0, (0.0, 0.0, 0.0), 0.0)]
    from paper_2503_08217_gb300.render import Renderer
    r = Renderer(n, n_inst, cams)
    grads = {"means": _cu(gm), "quats": _cu(gq), "sh": _cu(gs),
             "inst_quat": torch.full((n_inst, 4), float("nan"), device="cuda"),
             "inst_trans": torch.full((n_inst, 3), float("nan"), device="cuda")}
    r.ws.to_world_bwd(cs, poses, grads)
    torch.cuda.synchronize()
    for name, b in (("means", e_m), ("quats", e_q), ("sh", e_s), ("inst_quat", e_pq), ("inst_trans", e_pt)):
        a = grads[name].double().cpu().numpy()
        assert _rel(a, b) <= 1e-4, (name, _rel(a, b))
        if name.startswith("inst"):
            assert (a[[1, 5]] == 0).all()                   # empty instances


# ----------------------------------------------------- record and selection
# pairs of Gaussians by 128-bit accesses where both arrays are 16-byte aligned,
# one by one from an odd start; 2,048 Gaussians a block
@pytest.mark.parametrize("n", [1, 2, 31, 33, 2047, 2049, 4100])
@pytest.mark.parametrize("start", [(0, 0), (1, 1), (0, 1)])
def test_visibility_record_sub_ranges(n, start):
    from paper_2503_08217_gb300 import binding
    rng = np.random.default_rng(n)
    life = rng.uniform(-1, 1, (n + 2, 2)).astype(np.float32)
    vis = rng.uniform(-1, 1, (n + 2, 2)).astype(np.float32)
    seen = rng.random(n) < 0.5
    bits = np.packbits(np.r_[seen, np.zeros(-n % 32, bool)], bitorder="little").view(np.int32)
    t = np.float32(0.25)
    for mode in (binding.VIS_RECORD, binding.VIS_FINALIZE, binding.VIS_RESET):
        dl, dv, mask = _cu(life), _cu(vis), _cu(bits)
        a, b = start
        binding.update_visibility(n, float(t), mask if mode == binding.VIS_RECORD else None,
                                  dl[a:a + n], dv[b:b + n], mode)
        want_l, want_v = life.copy(), vis.copy()
        part = want_l[a:a + n].copy()
        if mode == binding.VIS_RECORD:
            oracle.vis_record(part, seen, t)
            want_l[a:a + n] = part
        elif mode == binding.VIS_FINALIZE:
            want_v[b:b + n] = oracle.vis_finalize(part)
        else:
            want_v[b:b + n], want_l[a:a + n] = oracle.vis_reset(n)
        np.testing.assert_array_equal(dl.cpu().numpy(), want_l)
        np.testing.assert_array_equal(dv.cpu().numpy(), want_v)


def test_static_selection_in_turn():
    """One scratch for all calls: sizes up and down, empty ones between them."""
    from paper_2503_08217_gb300 import binding
    rng = np.random.default_rng(31)
    for n in (4097, 0, 1, 70_001, 4096, 0, 70_001, 33):
        vis = np.sort(rng.uniform(-1, 1, (n, 2)).astype(np.float32), axis=1)
        idx = torch.full((max(n, 1),), -1, dtype=torch.int32, device="cuda")
        count = torch.full((1,), -7, dtype=torch.int32, device="cuda")
        binding.select_visible_static(_cu(vis), 0.1, idx, count)
        want = oracle.select(vis, 0.1) if n else np.zeros(0, np.int64)
        assert int(count.item()) == want.size
        np.testing.assert_array_equal(idx[:want.size].cpu().numpy(), want)


# ------------------------------------------------------------- render routes
def _step(scene, cams, vis, dL, step=3, **kw):
    import gpu_helpers
    return gpu_helpers.gpu_step(scene, step, cams, vis, dL=dL, **kw)


@pytest.fixture(scope="module")
def tiny():
    import gpu_helpers
    scene = scenegen.generate("tiny", seed=0)
    return scene, gpu_helpers.sweep_visibility(scene)[0]


def test_forward_warps_per_tile_agree(tiny):
    """Copies of one camera on both sides of the tile count from which two warps
    walk a tile instead of four: the same pixels, last contributors and
    transmittances, and gradients in proportion to the copies."""
    scene, vis = tiny
    cam = scene.cams[3][0]
    tiles = ((cam.width + 15) // 16) * ((cam.height + 15) // 16)
    line = torch.cuda.get_device_properties(0).multi_processor_count * 18
    few = min(line // tiles, 31)
    assert few >= 1 and (few + 1) * tiles > line, "the line is out of reach of 32 views"
    d = np.random.default_rng(37).standard_normal((3, cam.height, cam.width))
    kw = {"max_splats": scene.n * (few + 1), "max_duplicates": 8 * scene.n * (few + 1)}
    out = []
    for copies in (few, few + 1):
        res = _step(scene, [cam] * copies, vis, [d / copies] * copies, **kw)
        P = cam.width * cam.height
        for v in range(1, copies):
            np.testing.assert_array_equal(res["images"][v], res["images"][0])
            np.testing.assert_array_equal(res["n_contrib"][v * P:(v + 1) * P], res["n_contrib"][:P])
        out.append((res["images"][0], res["n_contrib"][:P], res["final_T"][:P], res["grads"]))
    (ia, na, ta, ga), (ib, nb, tb, gb) = out
    np.testing.assert_allclose(ia, ib, rtol=0, atol=1e-6)
    np.testing.assert_array_equal(na, nb)
    np.testing.assert_allclose(ta, tb, rtol=0, atol=1e-6)
    _close_grads(ga, gb)


@pytest.mark.parametrize("extra", [0, 1])
def test_overlapped_and_plain_launches_agree(tiny, extra):
    """A scene padded with never-visible static Gaussians to the size up to
    which launches overlap, and to one more, renders and differentiates as the
    scene alone does."""
    scene, vis = tiny
    pad = 2_000_000 + extra - scene.n
    big = copy.deepcopy(scene)
    s = int(scene.inst_offsets[1])
    for k in ("means", "log_scales", "quats", "opacity_logits", "sh"):
        a = getattr(scene, k)
        fill = np.zeros((pad,) + a.shape[1:], a.dtype)
        if k == "quats":
            fill[:, 0] = 1
        setattr(big, k, np.concatenate([a[:s], fill, a[s:]]))
    big.inst_offsets = scene.inst_offsets.copy()
    big.inst_offsets[1:] += pad
    never = np.tile(np.array([[0.9, -0.9]], np.float32), (pad, 1))
    cams = scene.cams[3]
    d = [np.random.default_rng(41).standard_normal((3, c.height, c.width)) for c in cams]
    a = _step(scene, cams, vis, d)
    b = _step(big, cams, np.concatenate([vis[:s], never, vis[s:]]), d,
              max_splats=a["renderer"].ws.capacity.max_splats)
    assert big.means.shape[0] == 2_000_000 + extra
    for x, y in zip(a["images"], b["images"]):
        np.testing.assert_allclose(x, y, rtol=0, atol=1e-6)
    g = {}
    for k in NAMES:
        q = b["grads"][k]
        if not k.startswith("inst"):
            assert not q[s:s + pad].any(), k
            q = np.concatenate([q[:s], q[s + pad:]])
        g[k] = q
    _close_grads(g, a["grads"])


@pytest.mark.parametrize("count,width,height", [(1, 640, 1600), (40, 640, 1600), (40, 2000, 48), (300, 33, 600)])
def test_expansion_of_tall_and_wide_splats(count, width, height):
    """Splats of up to 100 tile rows (more than a warp's lanes) and 4,000 tiles
    (more than a chunk of pairs), chunk boundaries inside rows."""
    import gpu_helpers
    from test_gpu_parity import _stage_isolated_sort
    rng = np.random.default_rng(count)
    g = scenegen.generate("fd", seed=2, n_static=count, n_inst=0, n_steps=2)
    g.means[:] = rng.uniform((-1, -1, 4), (1, 1, 8), (count, 3))
    g.log_scales[:] = np.log(rng.uniform(0.05, 4.0, (count, 3)))
    g.log_scales[0] = np.log(4.0)
    g.opacity_logits[:] = rng.uniform(-1, 3, g.opacity_logits.shape)
    cams = [make_camera(width, height, 300.0, (0.0, 0.0, 0.0), 0.0)]
    g = scenegen.with_cameras(g, [cams, cams])
    tiles = ((width + 15) // 16) * ((height + 15) // 16)
    for rows in (0, 1):                                     # 1: nearly every splat overflows the row table
        r = gpu_helpers.Renderer(g.n, 0, cams, max_duplicates=max(4096, count * tiles), max_rows=rows)
        res = _step(g, cams, oracle.vis_reset(count)[0], None, step=0, renderer=r)
        assert res["counts"]["n_duplicates"] >= tiles // 4
        _stage_isolated_sort(res, cams)


@pytest.mark.parametrize("width,height", [(32, 16), (128, 128), (80, 208), (2048, 2048), (2064, 2048)])
def test_sort_at_short_tile_digits(width, height):
    """2, 64, 65, 16,384 and 16,512 tiles: both sides of the lines (6 bits of the
    first and of the second digit) between the two ways of ranking a digit."""
    import gpu_helpers
    from test_gpu_parity import _stage_isolated_sort
    rng = np.random.default_rng(53)
    count = 600
    g = scenegen.generate("fd", seed=3, n_static=count, n_inst=0, n_steps=2)
    g.means[:] = rng.uniform((-3, -3, 3), (3, 3, 9), (count, 3))
    g.log_scales[:] = np.log(rng.uniform(0.01, 0.1, (count, 3)))
    cams = [make_camera(width, height, 0.5 * max(width, height), (0.0, 0.0, 0.0), 0.0)]
    g = scenegen.with_cameras(g, [cams, cams])
    r = gpu_helpers.Renderer(g.n, 0, cams, max_duplicates=1 << 20)
    res = _step(g, cams, oracle.vis_reset(count)[0], None, step=0, renderer=r)
    assert res["counts"]["n_duplicates"] > count // 4
    _stage_isolated_sort(res, cams)


@pytest.mark.parametrize("n_inst", [40, 260])
def test_pose_sums_with_many_instances(tiny, n_inst):
    """Empty instances after the scene's own: fewer copies of the pose sums (64
    with up to 512 matrices, 20 at 6 x 261, near the most a call takes) give the
    same gradients, and an empty instance's are zero; also when added to."""
    import gpu_helpers
    from paper_2503_08217_gb300.render import DeviceScene
    scene, vis = tiny
    cams = [scene.cams[3][0]] * 6
    more = copy.deepcopy(scene)
    extra = n_inst - scene.n_inst
    more.inst_offsets = np.r_[scene.inst_offsets, np.full(extra, scene.n)].astype(np.int64)
    more.inst_quat = np.concatenate([scene.inst_quat, np.tile(np.array([1, 0, 0, 0], np.float32),
                                                              (scene.n_steps, extra, 1))], 1)
    more.inst_trans = np.concatenate([scene.inst_trans, np.zeros((scene.n_steps, extra, 3), np.float32)], 1)
    d = [np.random.default_rng(43).standard_normal((3, c.height, c.width)) for c in cams]
    kw = {"max_splats": 6 * scene.n, "max_duplicates": 48 * scene.n}
    a = _step(scene, cams, vis, d, **kw)
    b = _step(more, cams, vis, d, **kw)
    g = dict(b["grads"])
    for k in ("inst_quat", "inst_trans"):
        assert not g[k][scene.n_inst:].any(), k
        g[k] = g[k][:scene.n_inst]
    _close_grads(g, a["grads"])
    # a second backward adds the same again: the sums were cleared in between
    r, dev = b["renderer"], DeviceScene.from_host(more)
    acc = {k: _cu(b["grads"][k].astype(np.float32)) for k in NAMES}
    dL = _cu(np.concatenate([x.reshape(-1) for x in d]).astype(np.float32))
    r.backward(dev, _cu(more.inst_quat[3]), _cu(more.inst_trans[3]), torch.zeros(3, device="cuda"), dL, acc)
    torch.cuda.synchronize()
    _close_grads({k: 0.5 * v.double().cpu().numpy() for k, v in acc.items()}, b["grads"])


def test_backward_in_threads_of_unlike_scenes():
    """Two threads, one with few instances and one with many (the backward's
    shared memory grows with them), each on its own workspace and stream: one
    thread's smaller request does not lower the limit under the other's."""
    import threading
    from test_gpu_parity import _rig_crop
    scene = _rig_crop()                                     # SH degree 3: 53 KB for the rows alone
    vis = oracle.vis_reset(scene.n)[0]
    cams = scene.cams[3]
    more = copy.deepcopy(scene)
    extra = 500
    more.inst_offsets = np.r_[scene.inst_offsets, np.full(extra, scene.n)].astype(np.int64)
    more.inst_quat = np.concatenate([scene.inst_quat, np.tile(np.array([1, 0, 0, 0], np.float32),
                                                              (scene.n_steps, extra, 1))], 1)
    more.inst_trans = np.concatenate([scene.inst_trans, np.zeros((scene.n_steps, extra, 3), np.float32)], 1)
    d = [np.random.default_rng(47).standard_normal((3, c.height, c.width)) for c in cams]
    want = _step(scene, cams, vis, d)["grads"]
    got, errors = {}, []

    def run(name, sc):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(3):
                    got[name] = _step(sc, cams, vis, d)["grads"]
        except Exception as e:   # noqa: BLE001  (reported by the main thread)
            errors.append((name, e))

    threads = [threading.Thread(target=run, args=a) for a in (("few", scene), ("many", more))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for name in ("few", "many"):
        g = {k: (v[:scene.n_inst] if k.startswith("inst") else v) for k, v in got[name].items()}
        _close_grads(g, want)
