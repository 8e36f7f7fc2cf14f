"""The workloads whose speed this framework is judged by.

Each case is a call sequence of a user's program: an image of a reconstruction
(``view``), a training step's forward and backward over one or several cameras
(``step``), a whole optimisation step (``train``), the optimiser alone
(``adam``), the visibility record's turn of an epoch (``record``), the
NeuralODE object poses (``ode``) and the conventional pipeline's world
transform (``world``). Sizes are those of the repository's synthetic street
corridors (``paper_2503_08217_gb300/scenegen.py``), redrawn on the GPU from the
seed with the same distributions, and sizes between and around them.

``exact`` restates every path in float64 PyTorch from the definitions.
"""
import math
import random

import numpy as np
import torch

from paper_2503_08217_gb300 import binding, scenegen
from paper_2503_08217_gb300.render import DeviceScene, FusedAdam, Renderer, render
from paper_2503_08217_gb300.train import PARAM_NAMES, Trainer, TrainState

DEV = "cuda"
GRAD_NAMES = PARAM_NAMES + ("inst_quat", "inst_trans")


# ---------------------------------------------------------------- the cases
def _scene_case(name, kind, n_static, n_inst, per_inst, length, width, height, focal, views,
                sh_degree, lod, half_width=20.0, y_max=15.0, route="batched"):
    c = {"kind": kind, "n_static": n_static, "n_inst": n_inst, "per_inst": per_inst,
         "length": length, "half_width": half_width, "y_max": y_max, "width": width,
         "height": height, "focal": focal, "views": views, "sh_degree": sh_degree, "lod": lod,
         "route": route}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a small preview image (the tiny corridor): launches and latency count
        _scene_case("view_tiny", "view", 20_000, 2, 1000, 80.0, 320, 192, 250.0, 1, 0, 0.0,
                    half_width=40.0, y_max=8.0),
        # a training step on a crop with ragged tiles, through torch autograd
        _scene_case("step_tiny", "step", 20_011, 2, 997, 80.0, 317, 187, 250.0, 1, 1, 0.0,
                    half_width=40.0, y_max=8.0, route="autograd"),
        # gradients of two odd-sized cameras summed by one call per camera
        _scene_case("step_views", "step", 300_007, 5, 3001, 120.0, 1001, 563, 500.0, 2, 2, 0.5,
                    route="per_view"),
        # an evaluation image of the mid corridor at 1080p
        _scene_case("view_mid", "view", 1_000_000, 20, 5000, 300.0, 1920, 1080, 960.0, 1, 3, 1.0),
        # a training step on the mid corridor, through torch autograd
        _scene_case("step_mid", "step", 1_000_000, 20, 5000, 300.0, 1920, 1080, 960.0, 1, 3, 1.0,
                    route="autograd"),
        # an image of the large corridor at full detail (no LOD cull)
        _scene_case("view_large", "view", 8_000_000, 80, 12_500, 1500.0, 1920, 1280, 960.0, 1, 3,
                    0.0),
        # the surround rig: forward and backward of seven cameras in one call
        _scene_case("step_rig", "step", 8_000_000, 80, 12_500, 1500.0, 1920, 1080, 960.0, 7, 3, 1.0),
        # a whole optimisation step on the training corridor, seven cameras
        _scene_case("train_rig", "train", 16_000_000, 120, 12_500, 2000.0, 1920, 1080, 960.0, 7, 3,
                    1.0),
        # the optimiser over the mid corridor's parameters
        {"name": "adam_mid", "kind": "adam", "n": 1_100_003, "sh_degree": 3},
        # the end of an epoch at the large corridor: last frustum mask, windows, selection
        {"name": "record_large", "kind": "record", "n": 9_000_001},
        # poses of the training corridor's instances over its timesteps, with the reverse mode
        {"name": "ode_train", "kind": "ode", "n_inst": 120, "n_times": 400, "substeps": 2, "embed": 8},
        # moving the large corridor's instances to the world frame, and the adjoints back
        {"name": "world_large", "kind": "world", "n_static": 1000, "n_inst": 80, "per_inst": 12_500,
         "sh_degree": 3},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["view", "view", "step", "step", "step", "train", "adam", "record", "ode",
                       "world"])
    if kind == "adam":
        return {"kind": kind, "n": log_int(1000, 4_000_000), "sh_degree": rng.randrange(4)}
    if kind == "record":
        return {"kind": kind, "n": log_int(1000, 16_000_000)}
    if kind == "ode":
        return {"kind": kind, "n_inst": log_int(1, 120), "n_times": log_int(2, 400),
                "substeps": rng.randint(1, 2), "embed": rng.choice([0, 3, 4, 8])}
    if kind == "world":
        return {"kind": kind, "n_static": log_int(1, 1000), "n_inst": log_int(1, 80),
                "per_inst": log_int(50, 12_500), "sh_degree": rng.randrange(4)}
    views = rng.choice([1, 1, 2, 3, 7])
    n = log_int(10_000, 8_000_000 if kind != "train" else 4_000_000)
    # the corridors' densities: 250 Gaussians per metre (tiny) to 5,333 (large)
    length = max(30.0, n / rng.uniform(250.0, 5333.0))
    width = rng.randint(200, 1920)
    height = rng.randint(int(0.5 * width), int(0.67 * width))
    return _scene_case(None, kind, n, rng.choice([0, 1, 5, 20, 80]), log_int(50, 5000), length,
                       width, height, width * rng.uniform(0.5, 0.8), views, rng.randrange(4),
                       rng.choice([0.0, 0.5, 1.0, 2.0]),
                       route=rng.choice(["batched", "autograd", "per_view"]) if kind == "step"
                       else "batched")


# ---------------------------------------------------------------- inputs
class _Draw:
    """Seeded draws on the GPU."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(int(seed))

    def uniform(self, lo, hi, *shape):
        return torch.empty(shape, device=DEV).uniform_(lo, hi, generator=self.g)

    def normal(self, *shape, std=1.0, mean=0.0):
        return torch.empty(shape, device=DEV).normal_(mean, std, generator=self.g)


def _rotations(d, n):
    q = d.normal(n, 4)
    return q / q.norm(dim=1, keepdim=True)


def _sh(d, n, degree):
    k = (degree + 1) ** 2
    sh = d.normal(n, k, 3, std=0.05)
    sh[:, 0] = d.uniform(-math.sqrt(math.pi), math.sqrt(math.pi), n, 3)
    return sh


def _instance_poses(d, n_inst, length):
    """Vehicles on the road: yawed by up to 0.1 rad, anywhere along the corridor."""
    yaw = d.uniform(-0.1, 0.1, n_inst)
    zero = torch.zeros_like(yaw)
    quat = torch.stack([torch.cos(0.5 * yaw), zero, torch.sin(0.5 * yaw), zero], 1).contiguous()
    trans = torch.stack([d.uniform(-8.0, 8.0, n_inst), torch.ones_like(yaw),
                         d.uniform(0.0, length, n_inst)], 1).contiguous()
    return quat, trans


def _corridor(case, d):
    """(scene, instance quaternions, instance translations): static Gaussians
    3x denser within 5 m of the road, instances in 2 x 2 x 4 m boxes."""
    ns, nd = case["n_static"], case["n_inst"] * case["per_inst"]
    n = ns + nd
    means = torch.empty(n, 3, device=DEV)
    means[:ns, 0] = d.uniform(-case["half_width"], case["half_width"], ns)
    low, high = 3.0 * 7.0, case["y_max"] - 5.0
    dense = d.uniform(0.0, 1.0, ns) < low / (low + high)
    means[:ns, 1] = torch.where(dense, d.uniform(-2.0, 5.0, ns), d.uniform(5.0, case["y_max"], ns))
    means[:ns, 2] = d.uniform(0.0, case["length"], ns)
    means[ns:, :2] = d.uniform(-1.0, 1.0, nd, 2)
    means[ns:, 2] = d.uniform(-2.0, 2.0, nd)
    off = torch.tensor([0] + [ns + k * case["per_inst"] for k in range(case["n_inst"] + 1)],
                       dtype=torch.int64, device=DEV)
    scene = DeviceScene(means=means, log_scales=d.normal(n, 3, std=0.5, mean=-2.0),
                        quats=_rotations(d, n), opacity_logits=d.normal(n),
                        sh=_sh(d, n, case["sh_degree"]), inst_offsets=off,
                        sh_degree=case["sh_degree"])
    return (scene,) + _instance_poses(d, case["n_inst"], case["length"])


def _rig(case):
    """The cameras at the middle of the corridor; a rig's cameras past the
    fifth are smaller, as on the surround rig."""
    pos, n = (0.0, 0.0, 0.5 * case["length"]), case["views"]
    cams = []
    for k in range(n):
        w, h, f = case["width"], case["height"], case["focal"]
        if k >= 5:
            w, h, f = 2 * w // 3, 8 * h // 9, 2.0 * f / 3.0
        cams.append(scenegen.make_camera(w, h, f, pos, 2.0 * math.pi * k / n))
    return cams


def _record(case, scene):
    """The visibility record after the first epoch at rendering time 0: a front
    camera sees a Gaussian until it has passed it, a surround rig always; the
    instances move with the traffic and are seen throughout."""
    n, ns = scene.n, case["n_static"]
    life = torch.empty(n, 2, device=DEV)
    life[:, 0] = -1.0
    life[:, 1] = 1.0
    if case["views"] < 3:
        life[:ns, 1] = 2.0 * scene.means[:ns, 2] / case["length"] - 1.0
    window = torch.empty_like(life)
    window[:, 0] = life[:, 0] - 0.1
    window[:, 1] = life[:, 1] + 0.1
    return window, life


def _scene_inputs(case, seed):
    d = _Draw(seed)
    scene, quat, trans = _corridor(case, d)
    cams = _rig(case)
    window, life = _record(case, scene)
    pixels = sum(c.width * c.height for c in cams)
    d_image = d.normal(3 * pixels, std=1.0 / pixels)
    background = d.uniform(0.0, 1.0, 3)
    return scene, quat, trans, cams, window, life, d_image, background


def _param_sizes(n, degree):
    return [(n, 3), (n, 3), (n, 4), (n,), (n, (degree + 1) ** 2, 3)]


def _adam_inputs(case, seed):
    """Parameters, gradients and moments of a run in progress (after 100 steps)."""
    d = _Draw(seed)
    shapes = _param_sizes(case["n"], case["sh_degree"])
    p = [d.normal(*s) for s in shapes]
    g = [d.normal(*s, std=1e-6) for s in shapes]
    m = [d.normal(*s, std=1e-6) for s in shapes]
    v = [d.normal(*s, std=1e-6).square_() for s in shapes]
    return p, g, m, v


def _record_inputs(case, seed):
    d = _Draw(seed)
    n = case["n"]
    mask = torch.randint(-2 ** 31, 2 ** 31, ((n + 31) // 32,), generator=d.g, device=DEV,
                         dtype=torch.int64).to(torch.int32)
    a, b = d.uniform(-1.0, 1.0, n), d.uniform(-1.0, 1.0, n)
    life = torch.stack([torch.minimum(a, b), torch.maximum(a, b)], 1).contiguous()
    return mask, life, float(np.float32(random.Random(seed).uniform(-0.9, 0.9)))


def _ode_inputs(case, seed):
    k, t = case["n_inst"], case["n_times"]
    params, embed, z0 = scenegen.ode_model(int(seed), k, max(1, case["embed"]))
    if case["embed"] == 0:
        h = 64
        params = np.concatenate([params[:8 * h].reshape(h, 8)[:, :7].reshape(-1), params[8 * h:]])
        embed = None
    cu = lambda a: None if a is None else torch.from_numpy(np.ascontiguousarray(a)).to(DEV)  # noqa: E731
    d = _Draw(seed)
    times = torch.from_numpy(np.linspace(-1.0, 1.0, t).astype(np.float32)).to(DEV)
    return (cu(params), cu(embed), cu(z0), times, d.normal(t, k, 4), d.normal(t, k, 3))


def _world_inputs(case, seed):
    d = _Draw(seed)
    c = dict(case, half_width=20.0, y_max=15.0, length=1500.0)
    scene, quat, trans = _corridor(c, d)
    up = [d.normal(*s) for s in _param_sizes(scene.n, case["sh_degree"])]
    return scene, quat, trans, {"means": up[0], "quats": up[2], "sh": up[4]}


def _capacities(n, cams):
    """Room for two views of every Gaussian; in small scenes close to the
    camera a splat covers tens of tiles."""
    splats = max(1024, n * min(len(cams), 2))
    return {"max_splats": splats, "max_duplicates": max(8 * splats, min(128 * splats, 1 << 25))}


# ---------------------------------------------------------------- prepare and run
def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind in ("view", "step", "train"):
        scene, quat, trans, cams, window, life, d_image, background = _scene_inputs(case, seed)
        s.update(scene=scene, quat=quat, trans=trans, cams=cams, window=window, life=life,
                 d_image=d_image, background=background)
        if kind == "train":
            s["trainer"], s["target"] = _trainer(case, seed, s)
            return s
        per_call = cams[:1] if case["route"] == "per_view" else cams
        s["renderer"] = Renderer(scene.n, scene.n_inst, per_call, **_capacities(scene.n, per_call))
        if kind == "step":
            tensors = scene.params() + [quat, trans]
            if case["route"] == "autograd":
                for t in tensors:
                    t.requires_grad_(True)
            else:
                s["grads"] = {k: torch.zeros_like(t) for k, t in zip(GRAD_NAMES, tensors)}
            if case["route"] == "per_view":
                s["d_images"] = list(torch.split(d_image, [3 * c.width * c.height for c in cams]))
    elif kind == "adam":
        p, g, m, v = _adam_inputs(case, seed)
        opt = FusedAdam(p, lr=1e-3)
        opt.exp_avg, opt.exp_avg_sq, opt.t = m, v, 100
        s.update(opt=opt, g=g)
    elif kind == "record":
        mask, life, t = _record_inputs(case, seed)
        n = case["n"]
        s.update(mask=mask, life=life, t=t, window=torch.zeros(n, 2, device=DEV),
                 idx=torch.zeros(n, dtype=torch.int32, device=DEV),
                 count=torch.zeros(1, dtype=torch.int32, device=DEV))
    elif kind == "ode":
        params, embed, z0, times, g_quat, g_trans = _ode_inputs(case, seed)
        s.update(params=params, embed=embed, z0=z0, times=times, g_quat=g_quat, g_trans=g_trans,
                 grads=[torch.zeros_like(params),
                        torch.zeros_like(embed) if embed is not None else None,
                        torch.zeros_like(z0)])
    else:
        scene, quat, trans, up = _world_inputs(case, seed)
        cam = scenegen.make_camera(16, 16, 16.0, (0.0, 0.0, 0.0), 0.0)
        s.update(scene=scene, up=up, c_scene=scene.c_scene(),
                 poses=binding.make_poses(quat, trans), held=(quat, trans),
                 ws=Renderer(scene.n, scene.n_inst, [cam], max_splats=1024, max_duplicates=4096).ws,
                 out=[scene.means.clone(), scene.quats.clone(), scene.sh.clone()],
                 grads={**{k: t.clone() for k, t in up.items()},
                        "inst_quat": torch.zeros_like(quat), "inst_trans": torch.zeros_like(trans)})
    return s


def _trainer(case, seed, s):
    """A trainer in the middle of a run: moments of 100 steps, one timestep's poses."""
    d = _Draw(seed + 1_000_003)
    state = TrainState.initial(s["scene"], s["quat"][None], s["trans"][None], s["window"], s["life"],
                               {"mode": "threshold", "r": case["lod"]})
    for m, v in zip(state.exp_avg + state.pose_exp_avg, state.exp_avg_sq + state.pose_exp_avg_sq):
        m.normal_(0.0, 1e-7, generator=d.g)
        v.normal_(0.0, 1e-6, generator=d.g).square_()
    state.adam_steps, state.pose_steps = 100, [100]
    trainer = Trainer(state, [s["cams"]], [0.0], background=s["background"],
                      **_capacities(s["scene"].n, s["cams"]))
    target = d.uniform(0.0, 1.0, s["d_image"].numel())
    return trainer, target


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "view":
        return {"image": s["renderer"].forward(s["scene"], s["quat"], s["trans"], s["cams"], 0.0,
                                               s["window"], None, case["lod"], s["background"])}
    if kind == "step":
        return _run_step(s, case)
    if kind == "train":
        loss, image = s["trainer"].step(0, s["target"], check=False)
        state = s["trainer"].state
        return {"loss": loss, "image": image, "life": s["life"],
                **{k: p for k, p in zip(PARAM_NAMES, state.scene.params())},
                "inst_quat": state.inst_quat, "inst_trans": state.inst_trans}
    if kind == "adam":
        s["opt"].step(s["g"])
        return s["opt"].params + s["opt"].exp_avg + s["opt"].exp_avg_sq
    if kind == "record":
        n, t = case["n"], s["t"]
        binding.update_visibility(n, t, s["mask"], s["life"], s["window"], binding.VIS_RECORD)
        binding.update_visibility(n, t, None, s["life"], s["window"], binding.VIS_FINALIZE)
        binding.select_visible_static(s["window"], t, s["idx"], s["count"])
        return {"life": s["life"], "window": s["window"], "idx": s["idx"], "count": s["count"]}
    if kind == "ode":
        states, quat, trans = binding.ode_poses(s["params"], s["embed"], s["z0"], s["times"],
                                                case["substeps"])
        for g in s["grads"]:
            if g is not None:
                g.zero_()
        binding.ode_poses_bwd(s["params"], s["embed"], s["times"], case["substeps"], states,
                              s["g_quat"], s["g_trans"], *s["grads"])
        return {"states": states, "quat": quat, "trans": trans, "grads": s["grads"]}
    # world: the render between the two calls writes the adjoints of the moved rows
    binding.to_world(s["c_scene"], s["poses"], *s["out"])
    g, first = s["grads"], case["n_static"]
    for k, up in s["up"].items():
        g[k][first:].copy_(up[first:])
    s["ws"].to_world_bwd(s["c_scene"], s["poses"], g)
    return {"moved": s["out"], "grads": g}


def _run_step(s, case):
    scene, quat, trans, r = s["scene"], s["quat"], s["trans"], s["renderer"]
    if case["route"] == "autograd":
        image = render(r, scene, s["cams"], 0.0, case["lod"], s["background"], s["window"],
                       s["life"], quat, trans)
        grads = torch.autograd.grad(image, scene.params() + [quat, trans], s["d_image"])
        return {"image": image, "life": s["life"], **dict(zip(GRAD_NAMES, grads))}
    if case["route"] == "batched":
        image = r.forward(scene, quat, trans, s["cams"], 0.0, s["window"], s["life"], case["lod"],
                          s["background"])
        r.backward(scene, quat, trans, s["background"], s["d_image"], s["grads"], overwrite=True)
        return {"image": image, "life": s["life"], **s["grads"]}
    images = []
    for g in s["grads"].values():
        g.zero_()
    for cam, d in zip(s["cams"], s["d_images"]):
        images.append(r.forward(scene, quat, trans, [cam], 0.0, s["window"], s["life"],
                                case["lod"], s["background"]))
        r.backward(scene, quat, trans, s["background"], d, s["grads"])
    return {"image": images, "life": s["life"], **s["grads"]}


# ---------------------------------------------------------------- work
def work(case):
    kind = case["kind"]
    if kind == "adam":
        # parameter, gradient and two moments read; parameter and moments written
        n = case["n"] * (11 + 3 * (case["sh_degree"] + 1) ** 2)
        return {"bytes": 28 * n, "flops": 12 * n}
    if kind == "record":
        # life read and written, window written, mask read, index list written
        return {"bytes": case["n"] * (16 + 8 + 0.125 + 2), "flops": 6 * case["n"]}
    if kind == "ode":
        # four evaluations of f per step forward; as many and their reverse backward
        macs = 64 * (7 + case["embed"]) + 64 * 64 + 6 * 64
        steps = case["n_inst"] * (case["n_times"] - 1) * case["substeps"]
        return {"bytes": steps * 24 * 2 + case["n_inst"] * case["n_times"] * 56,
                "flops": steps * 4 * macs * 2 * 4}
    if kind == "world":
        # mean, quaternion and SH read and written, each way
        k = (case["sh_degree"] + 1) ** 2
        n = case["n_inst"] * case["per_inst"]
        return {"bytes": n * 2 * 2 * 4 * (7 + 3 * k), "flops": n * 2 * (60 + 18 * k * k)}
    n = case["n_static"] + case["n_inst"] * case["per_inst"]
    floats = 11 + 3 * (case["sh_degree"] + 1) ** 2
    pixels = sum(c.width * c.height for c in _rig(case))
    size = n * (4 * floats + 8) + 12 * pixels
    # a pixel is opaque after some 80 splats; 17 operations forward, 42 backward
    ops = 17 * 80 * pixels + 100 * n
    if kind != "view":
        size += n * 4 * floats + 12 * pixels + 16 * n
        ops += 42 * 80 * pixels + 100 * n
    if kind == "train":
        size += 24 * n * floats + 12 * pixels
        ops += 12 * n * floats
    return {"bytes": size, "flops": ops}


# ---------------------------------------------------------------- float64 restatements
def exact(case, seed):
    kind = case["kind"]
    if kind in ("view", "step"):
        return _exact_render(case, seed)
    if kind == "train":
        return None     # a second pass starts from the first's parameters
    if kind == "adam":
        return _exact_adam(case, seed)
    if kind == "record":
        mask, life, t = _record_inputs(case, seed)
        n = case["n"]
        bit = (mask.long()[:, None] >> torch.arange(32, device=DEV)) & 1
        seen = bit.reshape(-1)[:n].bool()
        life = life.double()
        life = torch.where(seen[:, None], torch.stack([life[:, 0].clamp(max=t),
                                                       life[:, 1].clamp(min=t)], 1), life)
        window = life + torch.tensor([-0.1, 0.1], dtype=torch.float64, device=DEV)
        return {"life": life, "window": window, "idx": None, "count": None}
    if kind == "ode":
        return _exact_ode(case, seed)
    return _exact_world(case, seed)


def _exact_adam(case, seed):
    p, g, m, v = [[x.double() for x in part] for part in _adam_inputs(case, seed)]
    f = lambda x: float(np.float32(x))  # noqa: E731
    lr, b1, b2, eps, step = f(1e-3), f(0.9), f(0.999), f(1e-8), 101
    m = [b1 * a + (1 - b1) * x for a, x in zip(m, g)]
    v = [b2 * a + (1 - b2) * x * x for a, x in zip(v, g)]
    p = [a - lr * (x / (1 - b1 ** step)) / ((y / (1 - b2 ** step)).sqrt() + eps)
         for a, x, y in zip(p, m, v)]
    return p + m + v


def _rot64(q):
    w, x, y, z = (q / q.norm(dim=-1, keepdim=True)).unbind(-1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)],
                       -1).reshape(*q.shape[:-1], 3, 3)


def _basis64(d, degree):
    """Real spherical harmonics (orthonormal, Condon-Shortley sign) at unit directions."""
    x, y, z = d.unbind(-1)
    c = lambda a, b: math.sqrt(a / (b * math.pi))  # noqa: E731
    Y = [torch.full_like(x, 0.5 / math.sqrt(math.pi))]
    if degree >= 1:
        Y += [-c(3, 4) * y, c(3, 4) * z, -c(3, 4) * x]
    if degree >= 2:
        Y += [c(15, 4) * x * y, -c(15, 4) * y * z, c(5, 16) * (2 * z * z - x * x - y * y),
              -c(15, 4) * x * z, c(15, 16) * (x * x - y * y)]
    if degree >= 3:
        Y += [-c(35, 32) * y * (3 * x * x - y * y), c(105, 4) * x * y * z,
              -c(21, 32) * y * (4 * z * z - x * x - y * y),
              c(7, 16) * z * (2 * z * z - 3 * x * x - 3 * y * y),
              -c(21, 32) * x * (4 * z * z - x * x - y * y), c(105, 16) * z * (x * x - y * y),
              -c(35, 32) * x * (x * x - 3 * y * y)]
    return torch.stack(Y, -1)


def _splats64(case, cam, p, seg, quat, trans):
    """Position, conic, opacity, colour, depth, LOD scale, radius and frustum
    flag of the Gaussians p (float64, segment ids seg) in one camera (Eq. 1)."""
    V = torch.as_tensor(np.asarray(cam.world_to_cam, np.float64), device=DEV)
    Vr, Vt = V[:, :3], V[:, 3]
    eye = torch.eye(3, dtype=torch.float64, device=DEV)
    Pr = torch.cat([eye[None], _rot64(quat)], 0)
    Pt = torch.cat([torch.zeros(1, 3, dtype=torch.float64, device=DEV), trans], 0)
    A = Vr @ Pr
    centre = -(Pr.transpose(1, 2) @ (Pt + torch.linalg.solve(Vr, Vt))[..., None])[..., 0]
    A, d = A[seg], p["means"] - centre[seg]
    x, y, z = (A @ d[..., None])[..., 0].unbind(-1)
    near = z > float(np.float32(cam.near))
    z1 = torch.where(near, z, torch.ones_like(z))
    B = A @ (_rot64(p["quats"]) * torch.exp(p["log_scales"])[:, None, :])
    fx, fy = float(np.float32(cam.fx)), float(np.float32(cam.fy))
    limx, limy = 1.3 * 0.5 * cam.width / fx, 1.3 * 0.5 * cam.height / fy
    tx, ty = (x / z1).clamp(-limx, limx), (y / z1).clamp(-limy, limy)
    C0 = (fx / z1)[:, None] * (B[:, 0] - tx[:, None] * B[:, 2])
    C1 = (fy / z1)[:, None] * (B[:, 1] - ty[:, None] * B[:, 2])
    a, b, c = (C0 * C0).sum(1), (C0 * C1).sum(1), (C1 * C1).sum(1)
    det = (a + 0.3) * (c + 0.3) - b * b
    conic = torch.stack([(c + 0.3) / det, -b / det, (a + 0.3) / det], 1)
    uv = torch.stack([fx * x / z1 + cam.cx, fy * y / z1 + cam.cy], 1)
    unit = d / d.norm(dim=1, keepdim=True)
    rgb = (torch.einsum("nk,nkc->nc", _basis64(unit, case["sh_degree"]), p["sh"]) + 0.5).clamp(min=0.0)
    with torch.no_grad():
        mid = 0.5 * (a + c)
        sigma = torch.sqrt(mid + torch.sqrt((0.25 * (a - c) ** 2 + b * b).clamp(min=0.0)))
        mid = mid + 0.3
        radius = torch.ceil(3 * torch.sqrt(mid + torch.sqrt((mid * mid - det).clamp(min=0.1))))
        grid = torch.tensor([(cam.width + 15) // 16, (cam.height + 15) // 16], device=DEV)
        lo = torch.floor((uv - radius[:, None]) / 16).clamp(min=0.0)
        hi = torch.floor((uv + radius[:, None] + 15) / 16).clamp(min=0.0)
        lo, hi = torch.minimum(lo.long(), grid), torch.minimum(hi.long(), grid)
        inside = near & (det > 0) & ((hi - lo) > 0).all(1)
        # tiles whose pixels the alpha >= 1/255 ellipse's box can reach
        reach = torch.sqrt((2 * torch.log(255 * torch.sigmoid(p["opacity_logits"])).clamp(min=0.0))
                           [:, None] * torch.stack([a + 0.3, c + 0.3], 1)) + 0.5
        lo = torch.maximum(lo, torch.floor((uv - reach) / 16).long())
        hi = torch.minimum(hi, torch.floor((uv + reach) / 16).long() + 1)
    return uv, conic, torch.sigmoid(p["opacity_logits"]), rgb, z, sigma, inside, lo, hi


def _blend64(cam, uv, conic, opac, rgb, z, lo, hi, background, d_image):
    """Eq. 2 over every tile; returns the image [3, H, W], and with d_image
    the adjoints of (uv, conic, opac, rgb)."""
    W, H = cam.width, cam.height
    gx, gy = (W + 15) // 16, (H + 15) // 16
    order = torch.argsort(z, stable=True)
    ext = (hi - lo).clamp(min=0)[order]
    count = ext[:, 0] * ext[:, 1]
    owner = torch.repeat_interleave(torch.arange(order.numel(), device=DEV), count)
    start = torch.cumsum(count, 0) - count
    k = torch.arange(owner.numel(), device=DEV) - start[owner]
    w = ext[owner, 0]
    tile = (lo[order][owner, 1] + torch.div(k, w, rounding_mode="floor")) * gx + lo[order][owner, 0] + k % w
    by_tile = torch.argsort(tile, stable=True)
    ids = order[owner[by_tile]]
    length = torch.bincount(tile, minlength=gx * gy)
    first = torch.cumsum(length, 0) - length
    tiles = torch.argsort(length)
    sizes = length[tiles].tolist()
    leaves = [t.detach().clone().requires_grad_(d_image is not None) for t in (uv, conic, opac, rgb)]
    image = torch.zeros(3, gy * 16, gx * 16, dtype=torch.float64, device=DEV)
    if d_image is not None:
        d_full = torch.zeros_like(image)
        d_full[:, :H, :W] = d_image.reshape(3, H, W)
    pix = torch.arange(256, device=DEV)
    at, budget = 0, 1 << 24
    while at < len(sizes):
        end = at + 1
        while end < len(sizes) and (end - at + 1) * 256 * sizes[end] <= budget:
            end += 1
        ts, L = tiles[at:end], max(1, sizes[end - 1])
        at = end
        px = (ts % gx)[:, None] * 16 + pix % 16
        py = torch.div(ts, gx, rounding_mode="floor")[:, None] * 16 + torch.div(pix, 16, rounding_mode="floor")
        slot = torch.arange(L, device=DEV)
        live = slot < length[ts][:, None]
        idx = ids[(first[ts][:, None] + slot).clamp(max=max(0, ids.numel() - 1))] if ids.numel() else None
        if idx is None:
            image[:, py, px] = background[:, None, None]
            continue
        with torch.enable_grad():
            u, q, o, col = (t[idx] for t in leaves)                       # [t, L, ...]
            dx = u[:, None, :, 0] - (px[:, :, None] + 0.5)
            dy = u[:, None, :, 1] - (py[:, :, None] + 0.5)
            power = -0.5 * (q[:, None, :, 0] * dx * dx + q[:, None, :, 2] * dy * dy) \
                - q[:, None, :, 1] * dx * dy
            alpha = (o[:, None] * torch.exp(power)).clamp(max=0.99)
            with torch.no_grad():
                on = live[:, None] & (power <= 0) & (alpha >= 1.0 / 255.0)
                on &= torch.cumprod(torch.where(on, 1 - alpha, 1.0), 2) >= 1e-4
            alpha = torch.where(on, alpha, 0.0)
            after = torch.cumprod(1 - alpha, 2)
            before = torch.cat([torch.ones_like(after[..., :1]), after[..., :-1]], 2)
            out = torch.einsum("tpl,tlc->tpc", alpha * before, col) + after[..., -1:] * background
        if d_image is not None:
            out.backward(d_full[:, py, px].permute(1, 2, 0))
        image[:, py, px] = out.detach().permute(2, 0, 1)
    return image[:, :H, :W], [t.grad if t.grad is not None else torch.zeros_like(t) for t in leaves]


@torch.no_grad()
def _exact_render(case, seed):
    scene, quat, trans, cams, window, life, d_image, background = _scene_inputs(case, seed)
    step = case["kind"] == "step"
    n = scene.n
    background = background.double()
    selected = torch.nonzero((window[:, 0] <= 0.0) & (window[:, 1] >= 0.0)).flatten()
    segment = (torch.bucketize(selected, scene.inst_offsets[1:-1], right=True)
               if case["n_inst"] else torch.zeros_like(selected))
    quat, trans = quat.double(), trans.double()
    params = dict(zip(PARAM_NAMES, scene.params()))
    grads = {k: torch.zeros(v.shape, dtype=torch.float64, device=DEV) for k, v in params.items()}
    g_quat, g_trans = torch.zeros_like(quat), torch.zeros_like(trans)
    seen = torch.zeros(n, dtype=torch.bool, device=DEV)
    images, at = [], 0
    for cam in cams:
        keep = []
        for ids, seg in zip(selected.split(1 << 20), segment.split(1 << 20)):
            p = {k: v[ids].double() for k, v in params.items()}
            *_, sigma, inside, _, _ = _splats64(case, cam, p, seg, quat, trans)
            seen[ids[inside]] = True
            keep.append(torch.stack([ids, seg], 1)[inside & (sigma >= case["lod"])])
        ids, seg = torch.cat(keep).unbind(1) if keep else (selected, segment)
        p = {k: v[ids].double().requires_grad_(step) for k, v in params.items()}
        poses = [quat.clone().requires_grad_(step), trans.clone().requires_grad_(step)]
        with torch.enable_grad():
            uv, conic, opac, rgb, z, _, _, lo, hi = _splats64(case, cam, p, seg, *poses)
        size = 3 * cam.width * cam.height
        image, g = _blend64(cam, uv, conic, opac, rgb, z, lo, hi, background,
                            d_image[at:at + size].double() if step else None)
        images.append(image.reshape(-1))
        at += size
        if step and ids.numel():
            torch.autograd.backward([uv, conic, opac, rgb], g)
            for k in p:
                if p[k].grad is not None:
                    grads[k].index_add_(0, ids, p[k].grad)
            for total, t in zip((g_quat, g_trans), poses):
                if t.grad is not None:
                    total += t.grad
    if not step:
        return {"image": torch.cat(images)}
    life = life.double()
    life[:, 0] = torch.where(seen, life[:, 0].clamp(max=0.0), life[:, 0])
    life[:, 1] = torch.where(seen, life[:, 1].clamp(min=0.0), life[:, 1])
    return {"image": images if case["route"] == "per_view" else torch.cat(images), "life": life,
            **grads, "inst_quat": g_quat, "inst_trans": g_trans}


def _exact_ode(case, seed):
    params, embed, z0, times, g_quat, g_trans = _ode_inputs(case, seed)
    if (case["n_times"] - 1) * case["substeps"] > 1000:
        return None
    D, H = case["embed"], 64
    leaf = lambda t: t.double().requires_grad_(True)  # noqa: E731
    p, z0 = leaf(params), leaf(z0)
    e = leaf(embed) if embed is not None else None
    W1, b1, W2, b2, W3, b3 = torch.split(p, [H * (7 + D), H, H * H, H, 6 * H, 6])
    W1, W2, W3 = W1.view(H, 7 + D), W2.view(H, H), W3.view(6, H)
    bias = b1 if e is None else b1 + e @ W1[:, 7:].T

    def f(z, t):
        h = torch.tanh(z @ W1[:, :6].T + (t * W1[:, 6] + bias))
        return torch.addmm(b3, torch.tanh(torch.addmm(b2, h, W2.T)), W3.T)

    t32 = times.cpu().numpy()
    z, states, posed = z0, [z0], [z0]
    for j in range(case["n_times"] - 1):
        t0, h = float(t32[j]), (float(t32[j + 1]) - float(t32[j])) / case["substeps"]
        for i in range(case["substeps"]):
            t = t0 + i * h
            k1 = f(z, t)
            k2 = f(z + 0.5 * h * k1, t + 0.5 * h)
            k3 = f(z + 0.5 * h * k2, t + 0.5 * h)
            k4 = f(z + h * k3, t + h)
            z = z + (h / 6.0) * (k1 + 2 * k2 + 2 * k3 + k4)
            states.append(z)
        posed.append(z)
    posed = torch.stack(posed)
    r = posed[..., 3:]
    th = r.norm(dim=-1, keepdim=True)
    small = th < 1e-6
    safe = torch.where(small, torch.ones_like(th), th)
    quat = torch.cat([torch.where(small, 1 - (r * r).sum(-1, keepdim=True) / 8, torch.cos(0.5 * safe)),
                      torch.where(small, 0.5 * torch.ones_like(th), torch.sin(0.5 * safe) / safe) * r], -1)
    trans = posed[..., :3]
    leaves = [p] + ([e] if e is not None else []) + [z0]
    g = list(torch.autograd.grad([quat, trans], leaves, [g_quat.double(), g_trans.double()]))
    if e is None:
        g.insert(1, None)
    return {"states": torch.stack(states).detach(), "quat": quat.detach(), "trans": trans.detach(),
            "grads": g}


def _exact_world(case, seed):
    scene, quat, trans, up = _world_inputs(case, seed)
    first, per, deg = case["n_static"], case["per_inst"], case["sh_degree"]
    K = (deg + 1) ** 2
    dyn = lambda t: t[first:].double().view(case["n_inst"], per, *t.shape[1:])  # noqa: E731
    means, quats, sh = (dyn(t).requires_grad_(True) for t in (scene.means, scene.quats, scene.sh))
    pq, pt = quat.double().requires_grad_(True), trans.double().requires_grad_(True)
    R = _rot64(pq)
    moved = torch.einsum("kij,knj->kni", R, means) + pt[:, None]
    a, b = (pq / pq.norm(dim=-1, keepdim=True))[:, None], quats / quats.norm(dim=-1, keepdim=True)
    aw, av, bw, bv = a[..., :1], a[..., 1:].expand(*b.shape[:-1], 3), b[..., :1], b[..., 1:]
    turned = torch.cat([aw * bw - (av * bv).sum(-1, keepdim=True),
                        aw * bv + bw * av + torch.linalg.cross(av, bv, dim=-1)], -1)
    # the rotated coefficients give, at every world direction, the colour of the object frame's
    d = torch.randn(256, 3, dtype=torch.float64, device=DEV,
                    generator=torch.Generator(device=DEV).manual_seed(1))
    d = d / d.norm(dim=1, keepdim=True)
    D = torch.linalg.pinv(_basis64(d, deg)) @ _basis64(torch.einsum("sj,kji->ksi", d, R), deg)
    spun = torch.einsum("kij,knjc->knic", D.reshape(-1, K, K), sh)
    g = torch.autograd.grad([moved, turned, spun], [means, quats, sh, pq, pt],
                            [dyn(up[k]) for k in ("means", "quats", "sh")], allow_unused=True)

    def whole(static, part):
        return torch.cat([static[:first].double(), part.detach().reshape(-1, *static.shape[1:])])

    return {"moved": [whole(scene.means, moved), whole(scene.quats, turned), whole(scene.sh, spun)],
            "grads": {"means": whole(up["means"], g[0]), "quats": whole(up["quats"], g[1]),
                      "sh": whole(up["sh"], g[2]), "inst_quat": g[3], "inst_trans": g[4]}}
