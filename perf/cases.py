"""The work a user of the visibility cache has it do, as cases that can be timed.

Every case goes through the Python entry points of the package
(``paper_2506_05930_gb300.nvc``): whole frames, training steps, inference,
shading, clustered sampling, temporal resampling and the exact direct
illumination.  Networks and scenes are the repository's workloads (the tiny
float32 scene, the 1080p frame with 32 lights, online training, the four-view
frame with 128 lights, the 4K frame with 256 lights, the clustered cache and
the paper's preset), made here from a seed on the GPU.

The caches stand as a program has them in the middle of a run: 500 updates
done, Adam moments present for every table row that a lattice corner hashes
to (and zero for the rows none can reach), and the training frame number
advancing with every pass.
"""
import math

import numpy as np
import torch

from paper_2506_05930_gb300 import nvc

DEV = "cuda"
STEP0 = 500          # Adam updates a cache has behind it

# Hyper-parameters of the workloads' networks; `box` is the edge of the
# encoded domain, the rest are the library's configuration fields.
NETS = {
    "tiny": dict(n_levels=8, n_features=2, log2_table_size=14, base_resolution=4, growth=1.5,
                 hidden=(32, 32), leaky_slope=0.0, loss="l2", lr=1e-2, batch_positions=1024, box=1.0),
    "online": dict(n_levels=8, n_features=2, log2_table_size=14, base_resolution=4, growth=1.5,
                   hidden=(32, 32), leaky_slope=0.0, loss="bce", lr=1e-2, batch_positions=16384,
                   train_precision="fp16", loss_scale=128.0, box=1.0),
    "frame": dict(n_levels=16, n_features=2, log2_table_size=19, base_resolution=16, growth=1.447,
                  hidden=(64, 64, 64), leaky_slope=0.01, loss="bce", lr=1e-2, batch_positions=8192,
                  train_precision="fp16", loss_scale=128.0, box=10.0),
    "views": dict(n_levels=16, n_features=2, log2_table_size=19, base_resolution=16, growth=1.447,
                  hidden=(64, 64, 64), leaky_slope=0.01, loss="bce", lr=1e-2, batch_positions=8192,
                  train_precision="fp16", loss_scale=128.0, box=1.0),
    "sweep": dict(n_levels=16, n_features=2, log2_table_size=21, base_resolution=16, growth=1.447,
                  hidden=(64, 64, 64), leaky_slope=0.01, loss="bce", lr=1e-2, batch_positions=8192,
                  train_precision="fp32", box=10.0),
    "clustered": dict(n_levels=8, n_features=2, log2_table_size=19, base_resolution=2, growth=2.0,
                      hidden=(64, 64, 64), leaky_slope=0.01, loss="bce", lr=1e-2,
                      batch_positions=49152, train_precision="fp16", loss_scale=128.0, box=10.0),
    "paper": dict(n_levels=10, n_features=4, log2_table_size=14, base_resolution=16, growth=1.5,
                  hidden=(32, 32), leaky_slope=0.01, loss="l2", lr=0.05, lr_schedule="paper_ramp",
                  lr_end=1e-3, lr_ramp_steps=200, batch_positions=8192, box=10.0),
}
BETA1, BETA2, EPS = 0.9, 0.99, 1e-15
OUTS = ("idx", "pdf", "wsum", "radiance")


def listed():
    return [
        # the plain float32 path at its smallest: a 64x64 view of a scene with
        # four lights, training step and shading as one frame (launch-bound)
        dict(name="tiny_frame", kind="frame", net="tiny", lights=4, spheres=4, boxes=0,
             width=64, height=64, batch=1024, precision="fp32", table="fp32", tuned=False),
        # a probe query: visibilities at a thousand points, one fused launch
        dict(name="infer_probes", kind="infer", net="frame", lights=32, width=1000, height=1,
             precision="fp16", table="fp16", tuned=False),
        # online training of a small cache, tensor cores, 65,536 targets a step
        dict(name="online_step", kind="step", net="online", lights=4, spheres=4, boxes=0,
             width=64, height=64, batch=16384, precision="fp16", table="fp32"),
        # the paper's preset trained in float32
        dict(name="paper_step", kind="step", net="paper", lights=32, spheres=32, boxes=32,
             width=480, height=270, batch=8192, precision="fp32", table="fp32"),
        # the headline frame: training step, then inference + sampling + Neural DI
        dict(name="frame_1080p", kind="frame", net="frame", lights=32, spheres=32, boxes=32,
             width=1920, height=1080, batch=8192, precision="fp16", table="fp16", tuned=True),
        # shading alone at an odd window size and light count, bfloat16
        # operands, float32 table, the layout a program gets without tuning
        dict(name="shade_odd", kind="shade", net="frame", lights=21, width=1003, height=577,
             precision="bf16", table="fp32", tuned=False),
        # four views of one scene with 128 lights in one launch
        dict(name="multiview_128", kind="views", net="views", lights=128, width=3840, height=2160,
             precision="fp16", table="fp32", tuned=True),
        # many lights at 4K, half-precision table features
        dict(name="shade_4k_256", kind="shade", net="sweep", lights=256, width=3840, height=2160,
             precision="fp16", table="fp16", tuned=True),
        # the paper's preset on the float32 kernels at 1080p
        dict(name="paper_shade_fp32", kind="shade", net="paper", lights=32, width=1920, height=1080,
             precision="fp32", table="fp32", tuned=False),
        # a clustered frame: 1024 lights in 32 clusters, training step,
        # inference, two-step sampling with its shadow ray
        dict(name="clustered_1080p", kind="clustered", net="clustered", lights=1024, clusters=32,
             weights="sum", spheres=32, boxes=32, width=1920, height=1080, batch=49152,
             precision="fp16", table="fp16", tuned=True),
        # the cache as ReSTIR's candidate generator: sampling, temporal
        # merge with last frame's reservoirs, one shadow ray
        dict(name="restir_1080p", kind="restir", net="frame", lights=32, spheres=32, boxes=32,
             width=1920, height=1080, precision="fp16", table="fp16", tuned=True),
        # the reference picture: a shadow ray from every pixel to every light
        dict(name="exact_di_1080p", kind="exact_di", net="frame", lights=32, spheres=32, boxes=32,
             width=1920, height=1080),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: a kind of work, its sizes spread over its range."""
    kind = rng.choice(["tiny", "infer", "online", "paper_step", "frame", "shade", "views", "sweep",
                       "paper_shade", "clustered", "restir", "exact_di"])

    def view(hi):
        px = _log(rng, 64 * 64, hi)
        w = max(1, int(round(math.sqrt(px * rng.uniform(1.0, 2.4)))))
        return dict(width=w, height=max(1, px // w))

    def occluders(hi=48):
        return dict(spheres=rng.randint(1, hi), boxes=rng.randint(0, hi))

    low = rng.choice(["fp16", "bf16"])
    table = rng.choice(["fp16", "fp32"])
    if kind == "tiny":
        return dict(kind="frame", net="tiny", lights=rng.randint(1, 32), batch=_log(rng, 512, 8192),
                    precision="fp32", table="fp32", tuned=False, **occluders(16), **view(256 * 256))
    if kind == "infer":
        return dict(kind="infer", net="frame", lights=rng.randint(1, 40), width=_log(rng, 100, 2000000),
                    height=1, precision=low, table=table, tuned=False)
    if kind == "online":
        return dict(kind="step", net="online", lights=rng.randint(1, 32), batch=_log(rng, 1000, 32768),
                    precision=low, table="fp32", **occluders(16), **view(256 * 256))
    if kind == "paper_step":
        return dict(kind="step", net="paper", lights=rng.randint(8, 64), batch=_log(rng, 1000, 16384),
                    precision="fp32", table="fp32", **occluders(), **view(1920 * 1080))
    if kind == "frame":
        return dict(kind="frame", net="frame", lights=32, batch=8192, precision=low, table=table,
                    tuned=True, **occluders(), **view(2560 * 1440))
    if kind == "shade":
        prec = rng.choice(["fp16", "bf16", "fp8"])
        return dict(kind="shade", net="frame", lights=rng.randint(1, 48), precision=prec, table=table,
                    tuned=rng.random() < 0.5, **view(2560 * 1440))
    if kind == "views":
        return dict(kind="views", net="views", lights=rng.randint(64, 128), precision="fp16",
                    table="fp32", tuned=True, **view(3840 * 2160))
    if kind == "sweep":
        prec = rng.choice(["fp16", "bf16", "fp8"])
        return dict(kind="shade", net="sweep", lights=rng.randint(64, 256), precision=prec,
                    table="fp16", tuned=True, **view(3840 * 2160))
    if kind == "paper_shade":
        return dict(kind="shade", net="paper", lights=rng.randint(8, 64), precision="fp32",
                    table="fp32", tuned=False, **view(1920 * 1080))
    if kind == "clustered":
        return dict(kind="clustered", net="clustered", lights=_log(rng, 200, 2000),
                    clusters=rng.randint(8, 32), weights=rng.choice(["sum", "visibility"]),
                    batch=_log(rng, 8192, 49152), precision=low, table=table, tuned=True,
                    **occluders(), **view(1920 * 1080))
    if kind == "restir":
        return dict(kind="restir", net="frame", lights=rng.randint(8, 32), precision=low, table=table,
                    tuned=True, **occluders(), **view(2560 * 1440))
    return dict(kind="exact_di", net="frame", lights=rng.randint(4, 48), **occluders(64),
                **view(1920 * 1080))


# ------------------------------------------------------------ inputs --

def _gen(seed, salt):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 64 + salt)


def _rng(seed, salt):
    return np.random.Generator(np.random.PCG64([int(seed), salt]))


def _net(case):
    n = dict(NETS[case["net"]])
    box = n.pop("box")
    n.update(n_outputs=case.get("clusters") or case["lights"], precision=case.get("precision", "fp32"),
             table_precision=case.get("table", "fp32"), beta1=BETA1, beta2=BETA2, eps=EPS,
             bounds_min=(0.0, 0.0, 0.0), bounds_max=(box, box, box))
    if n["precision"] == "fp8":
        n["train_precision"] = "fp32"
    n.setdefault("train_precision", "fp32")
    n.setdefault("loss_scale", 1.0)
    n["batch_positions"] = case.get("batch", 1024)
    return n, box


def _resolutions(net):
    return [int(math.floor(net["base_resolution"] * net["growth"] ** l)) for l in range(net["n_levels"])]


def _hash(x, y, z, t):
    m = 0xFFFFFFFF
    return (x ^ ((y * 2654435761) & m) ^ ((z * 805459861) & m)) & (t - 1)


def _reached(net):
    """Per level the table rows that a corner of its lattice hashes to."""
    t = 1 << net["log2_table_size"]
    mask = torch.ones((net["n_levels"], t), device=DEV)
    for l, n in enumerate(_resolutions(net)):
        if (n + 1) ** 3 <= 4 * t:
            a = torch.arange(n + 1, device=DEV)
            rows = _hash(a.view(-1, 1, 1), a.view(1, -1, 1), a.view(1, 1, -1), t)
            mask[l] = 0.0
            mask[l, rows.reshape(-1)] = 1.0
    return mask


def _parameters(net, seed):
    """Parameters and Adam moments of a cache that has trained for a while."""
    g = _gen(seed, 1)
    f, t = net["n_features"], 1 << net["log2_table_size"]
    rows = _reached(net).unsqueeze(-1).expand(-1, -1, f).reshape(-1)
    n = rows.numel()
    parts = [0.15 * torch.randn(n, device=DEV, generator=g)]
    sm = [1e-5 * rows * torch.randn(n, device=DEV, generator=g)]
    sv = [rows * (1e-5 * (0.5 + torch.rand(n, device=DEV, generator=g))) ** 2]
    dims = [net["n_levels"] * f, *net["hidden"], net["n_outputs"]]
    for i, o in zip(dims[:-1], dims[1:]):
        parts.append(torch.randn(o * i, device=DEV, generator=g) * math.sqrt(2.0 / i))
        sm.append(1e-2 * torch.randn(o * i, device=DEV, generator=g))
        sv.append((1e-2 * (0.5 + torch.rand(o * i, device=DEV, generator=g))) ** 2)
    return torch.cat(parts), torch.cat(sm), torch.cat(sv)


def _view(case, box, seed, salt=0, width=None, height=None):
    """G-buffer: a heightfield with boxes seen from above (the 10-unit
    scenes) or points and normals at random (the unit-cube scenes)."""
    w, h = width or case["width"], height or case["height"]
    if box == 1.0:
        g = _gen(seed, 20 + salt)
        pos = torch.rand((w * h, 3), device=DEV, generator=g)
        nrm = torch.randn((w * h, 3), device=DEV, generator=g)
        return pos, torch.nn.functional.normalize(nrm, dim=1)
    r = _rng(seed, 40 + salt)
    a, fx, fy = r.uniform(0.1, 0.5, 8), r.uniform(0.3, 2.0, 8), r.uniform(0.3, 2.0, 8)
    px, py = r.uniform(0, 2 * np.pi, 8), r.uniform(0, 2 * np.pi, 8)
    x = ((torch.arange(w, device=DEV, dtype=torch.float64) + 0.5) / w * box).view(1, -1)
    y = ((torch.arange(h, device=DEV, dtype=torch.float64) + 0.5) / h * box).view(-1, 1)
    z = torch.full((h, w), 2.0, device=DEV, dtype=torch.float64)
    gx, gy = torch.zeros_like(z), torch.zeros_like(z)
    for k in range(8):
        sx, cx = torch.sin(fx[k] * x + px[k]), torch.cos(fx[k] * x + px[k])
        sy, cy = torch.sin(fy[k] * y + py[k]), torch.cos(fy[k] * y + py[k])
        z += a[k] * sx * sy
        gx += a[k] * fx[k] * cx * sy
        gy += a[k] * fy[k] * sx * cy
    for _ in range(16):
        c, s, top = r.uniform(0.5, 9.5, 2), r.uniform(0.2, 0.8, 2), r.uniform(2.0, 4.5)
        on = ((x - c[0]).abs() <= s[0]) & ((y - c[1]).abs() <= s[1]) & (z < top)
        z = torch.where(on, torch.full_like(z, top), z)
        gx, gy = gx.masked_fill(on, 0.0), gy.masked_fill(on, 0.0)
    nrm = torch.stack([-gx, -gy, torch.ones_like(z)], -1).reshape(-1, 3)
    pos = torch.stack([x.expand(h, w), y.expand(h, w), z], -1).reshape(-1, 3)
    return pos.float().contiguous(), torch.nn.functional.normalize(nrm, dim=1).float().contiguous()


def _scene_arrays(case, box, seed):
    """Lights, spheres and boxes; a clustered case has 16 rooms whose lights
    hang in fixtures and whose walls are boxes with doorways."""
    r = _rng(seed, 2)
    nl, ns, nb = case["lights"], case.get("spheres", 0), case.get("boxes", 0)
    if box == 1.0:
        lights = np.hstack([r.uniform(0, 1, (nl, 3)), r.uniform(0.5, 2.0, (nl, 1))])
        spheres = np.hstack([r.uniform(0, 1, (ns, 3)), r.uniform(0.05, 0.15, (ns, 1))])
        bc, bh = r.uniform(0, 1, (nb, 3)), r.uniform(0.02, 0.1, (nb, 3))
    else:
        lp = r.uniform(0, 10, (nl, 3))
        lp[:, 2] = r.uniform(4, 10, nl)
        lights = np.hstack([lp, r.uniform(20, 100, (nl, 1))])
        sc = r.uniform(0, 10, (ns, 3))
        sc[:, 2] = r.uniform(3, 9, ns)
        spheres = np.hstack([sc, r.uniform(0.2, 0.8, (ns, 1))])
        bc = r.uniform(0, 10, (nb, 3))
        bc[:, 2] = r.uniform(3, 9, nb)
        bh = r.uniform(0.2, 1.0, (nb, 3))
    boxes = np.hstack([bc - bh, bc + bh])
    if case["kind"] == "clustered":
        rooms, s = 4, 2.5
        fix = np.stack([np.repeat(np.arange(16), 2) % rooms, np.repeat(np.arange(16), 2) // rooms], 1) * s
        at = np.hstack([fix + r.uniform(0.3, s - 0.3, (32, 2)), r.uniform(7.0, 9.5, (32, 1))])
        g = r.integers(0, 32, nl)
        p = at[g] + r.normal(0.0, 0.15, (nl, 3))
        p[:, :2] = np.clip(p[:, :2], fix[g] + 0.1, fix[g] + s - 0.1)
        p[:, 2] = np.clip(p[:, 2], 4.0, 9.9)
        lights = np.hstack([p, r.uniform(20, 100, (nl, 1)) * 32.0 / nl])
        walls = []
        for i in range(1, rooms):
            for b in range(rooms):
                c, m = i * s, (b + 0.5) * s
                for lo, hi, z0 in ((b * s, m - 0.4, 0.0), (m + 0.4, (b + 1) * s, 0.0), (m - 0.4, m + 0.4, 5.0)):
                    walls.append([c - 0.04, lo, z0, c + 0.04, hi, 10.0])
                    walls.append([lo, c - 0.04, z0, hi, c + 0.04, 10.0])
        boxes = np.vstack([boxes, walls])
    return lights.astype(np.float32), spheres.astype(np.float32), boxes.astype(np.float32)


def _scene(case, box, seed):
    lights, spheres, boxes = _scene_arrays(case, box, seed)
    return nvc.Scene(lights, spheres, boxes, (0, 0, 0), (box, box, box))


def _views_of(case, box, seed):
    """The four views of a multi-view frame: the case's size and three smaller ones."""
    w, h = case["width"], case["height"]
    return [_view(case, box, seed, k, max(1, int(w * s)), max(1, int(h * s)))
            for k, s in enumerate((1 / 3, 1 / 2, 2 / 3, 1.0))]


def _outputs(n):
    return dict(idx=torch.empty(n, dtype=torch.int32, device=DEV), pdf=torch.empty(n, device=DEV),
                wsum=torch.empty(n, device=DEV), radiance=torch.empty(n, device=DEV))


def _clusters(case, scene_lights, seed):
    """k-means of the lights, as a program does once when it loads a scene."""
    init = _rng(seed, 3).choice(case["lights"], case["clusters"], replace=False).astype(np.int32)
    assign, _ = nvc.nvc_kmeans_lights(scene_lights, init, 10)
    return nvc.Clusters(assign, case["clusters"], weights=case["weights"]), assign


def prepare(case, seed):
    net, box = _net(case)
    kind = case["kind"]
    s = dict(case=case, seed=int(seed) & 0xFFFF, frame=0)
    if kind == "views":
        s["scene"] = _scene(case, box, seed)
        s["views"] = [nvc.View(p, n, k, **_outputs(p.shape[0]))
                      for k, (p, n) in enumerate(_views_of(case, box, seed))]
        big = s["views"][-1]
        s["pos"], s["nrm"] = big.pos, big.nrm
        out = {k: getattr(big, k) for k in OUTS}
    else:
        s["scene"] = _scene(case, box, seed)
        s["pos"], s["nrm"] = _view(case, box, seed)
        out = _outputs(s["pos"].shape[0])
    n = s["pos"].shape[0]
    s["out"] = out
    if kind == "exact_di":
        s["di"] = torch.empty(n, device=DEV)
        return s
    cache = s["cache"] = nvc.VisibilityCache(net, table_precision=net["table_precision"])
    s["h"] = cache.handle
    params, m, v = _parameters(net, seed)
    cache.set_params(params, m, v, step=STEP0)
    s["params"] = torch.empty_like(params)
    s["loss"] = torch.empty(1, dtype=torch.float64, device=DEV)
    if case.get("precision") == "fp8":
        nvc.nvc_calibrate(s["h"], s["pos"][:: max(1, n // 1024)][:1024].contiguous())
    if kind == "infer":
        s["vis"] = torch.empty((n, net["n_outputs"]), device=DEV)
    elif kind == "clustered":
        s["clusters"], s["assign"] = _clusters(case, _scene_arrays(case, box, seed)[0], seed)
        s["vis"] = torch.empty((n, net["n_outputs"]), device=DEV)
        s["light"] = torch.empty(n, dtype=torch.int32, device=DEV)
        s["weight"], s["estimate"] = torch.empty(n, device=DEV), torch.empty(n, device=DEV)
        nvc.nvc_autotune_infer(s["h"], s["pos"], s["vis"], reps=3)
    elif kind == "restir":
        g = _gen(seed, 5)
        s["light"] = [torch.randint(-1, case["lights"], (n,), device=DEV, generator=g, dtype=torch.int32),
                      torch.empty(n, dtype=torch.int32, device=DEV)]
        s["W"] = [30.0 * torch.rand(n, device=DEV, generator=g), torch.empty(n, device=DEV)]
        s["M"] = [torch.randint(0, 22, (n,), device=DEV, generator=g, dtype=torch.int32),
                  torch.empty(n, dtype=torch.int32, device=DEV)]
        s["cur_W"], s["estimate"] = torch.empty(n, device=DEV), torch.empty(n, device=DEV)
    if case.get("tuned") and kind != "clustered" and case["precision"] != "fp32":
        # as a program does once on its first frame
        nvc.nvc_autotune_shade_plan(s["h"], s["scene"], s["pos"], s["nrm"], reps=3, **out)
    return s


def run(s):
    case, f = s["case"], s["frame"]
    kind, seed = case["kind"], s["seed"]
    s["frame"] = f + 1
    if kind == "infer":
        nvc.nvc_infer(s["h"], s["pos"], s["vis"])
        return s["vis"]
    if kind == "shade":
        nvc.nvc_shade(s["h"], s["scene"], s["pos"], s["nrm"], seed, f,
                      fused=case["precision"] != "fp32", **s["out"])
        return s["out"]
    if kind == "exact_di":
        nvc.nvc_exact_di(s["scene"], s["pos"], s["nrm"], s["di"])
        return s["di"]
    if kind == "views":
        nvc.nvc_frame(s["h"], s["scene"], s["views"], nvc.NO_TRAINING, seed, f)
        return [{k: getattr(v, k) for k in OUTS} for v in s["views"]]
    if kind == "restir":
        a, b = f & 1, (f & 1) ^ 1
        nvc.nvc_wrs_sample(s["h"], s["scene"], s["pos"], s["nrm"], seed, f, idx=s["out"]["idx"],
                           pdf=s["out"]["pdf"], wsum=s["out"]["wsum"])
        torch.reciprocal(s["out"]["pdf"], out=s["cur_W"])
        nvc.nvc_temporal_merge(s["scene"], s["pos"], s["nrm"], s["out"]["idx"], s["cur_W"],
                               s["light"][a], s["W"][a], s["M"][a], seed, f, light=s["light"][b],
                               W=s["W"][b], M=s["M"][b], estimate=s["estimate"])
        return dict(idx=s["out"]["idx"], pdf=s["out"]["pdf"], wsum=s["out"]["wsum"],
                    light=s["light"][b], W=s["W"][b], M=s["M"][b], estimate=s["estimate"])
    if kind == "step":
        nvc.nvc_train_step(s["h"], s["scene"], s["pos"], seed, f, s["loss"])
        nvc.nvc_get_state(s["h"], s["params"])
        return dict(loss=s["loss"], params=s["params"])
    if kind == "frame":
        view = nvc.View(s["pos"], s["nrm"], 0, **s["out"])
        nvc.nvc_frame(s["h"], s["scene"], [view], 0, seed, f, s["loss"])
        nvc.nvc_get_state(s["h"], s["params"])
        return dict(loss=s["loss"], params=s["params"], **s["out"])
    nvc.nvc_train_step_clustered(s["h"], s["scene"], s["clusters"], s["pos"], seed, f, s["loss"])
    nvc.nvc_infer(s["h"], s["pos"], s["vis"])
    nvc.nvc_sample_clustered(s["scene"], s["clusters"], s["vis"], s["pos"], s["nrm"], seed, f,
                             light=s["light"], weight=s["weight"], estimate=s["estimate"])
    nvc.nvc_get_state(s["h"], s["params"])
    return dict(loss=s["loss"], params=s["params"], vis=s["vis"], light=s["light"],
                weight=s["weight"], estimate=s["estimate"])


# ------------------------------------------------------- least work --

def work(case):
    """Inputs read once, outputs written once; arithmetic counted from the
    method (a multiply-add as two)."""
    net, _ = _net(case)
    kind, L = case["kind"], case["lights"]
    lv, f, t = net["n_levels"], net["n_features"], 1 << net["log2_table_size"]
    px = case["width"] * case["height"]
    if kind == "views":
        px = sum(max(1, int(case["width"] * s)) * max(1, int(case["height"] * s))
                 for s in (1 / 3, 1 / 2, 2 / 3, 1.0))
    dims = [lv * f, *net["hidden"], net["n_outputs"]]
    macs = sum(a * b for a, b in zip(dims[:-1], dims[1:]))
    n_params = lv * t * f + macs
    # one entry per corner a pixel reads, never more than the table holds
    esize = 2 if case.get("table") == "fp16" else 4
    table = min(lv * t, 8 * lv * px) * f * esize + 4 * macs
    infer = 2 * macs + lv * (27 + 16 * f)
    occ = case.get("spheres", 0) + case.get("boxes", 0) + (72 if kind == "clustered" else 0)
    ray, light = 20 * occ + 20, 25
    b = fl = 0.0
    if kind in ("infer", "shade", "views", "frame", "restir", "clustered"):
        b += table + px * (12 if kind == "infer" else 24)
        fl += px * infer
    if kind in ("shade", "views", "frame"):
        b += 16 * px
        fl += px * L * (light + 10)
    if kind == "infer":
        b += 4 * L * px
    if kind == "restir":
        b += px * (12 + 12 + 16)
        fl += px * (L * (light + 10) + ray)
    if kind == "clustered":
        b += px * (4 * net["n_outputs"] + 12)
        fl += px * ((L * light if case["weights"] == "sum" else 0) + ray)
    if kind == "exact_di":
        return dict(bytes=28.0 * px, flops=float(px) * L * (light + ray))
    if kind in ("frame", "step", "clustered"):
        B = case["batch"]
        b += 28.0 * n_params + (2.0 * lv * t * f if esize == 2 else 0.0) + 4.0 * n_params
        fl += B * (3 * 2 * macs + 3 * lv * (27 + 16 * f)) + B * net["n_outputs"] * ray + 12.0 * n_params
    return dict(bytes=float(b), flops=float(fl))


# ------------------------------------------------ the values in 64 bits --

def _split(net, params):
    f, t = net["n_features"], 1 << net["log2_table_size"]
    n = net["n_levels"] * t * f
    dims = [net["n_levels"] * f, *net["hidden"], net["n_outputs"]]
    ws, off = [], n
    for i, o in zip(dims[:-1], dims[1:]):
        ws.append(params[off:off + i * o].view(o, i))
        off += i * o
    return params[:n].view(net["n_levels"], t, f), ws


def _logits64(net, box, params, pos):
    table, ws = _split(net, params)
    t = 1 << net["log2_table_size"]
    xh = (pos.double() / box).clamp(0.0, 1.0)
    feats = []
    for l, n in enumerate(_resolutions(net)):
        p = xh * n
        c = p.floor().clamp(max=n - 1)
        fr, c = p - c, c.long()
        e = 0.0
        for d in range(8):
            o = ((d & 1), (d >> 1) & 1, d >> 2)
            w = 1.0
            for k in range(3):
                w = w * (fr[:, k] if o[k] else 1.0 - fr[:, k])
            e = e + w.unsqueeze(1) * table[l][_hash(c[:, 0] + o[0], c[:, 1] + o[1], c[:, 2] + o[2], t)]
        feats.append(e)
    x = torch.cat(feats, 1)
    for k, w in enumerate(ws):
        x = x @ w.t()
        if k + 1 < len(ws):
            x = torch.where(x > 0, x, net["leaky_slope"] * x)
    return x


def _contributions64(pos, nrm, lights):
    d = lights[None, :, :3] - pos.double()[:, None, :]
    d2 = (d * d).sum(-1)
    cos = (d * nrm.double()[:, None, :]).sum(-1).clamp(min=0.0) / d2.sqrt()
    return lights[None, :, 3] * cos / (math.pi * d2.clamp(min=1e-6))


def _visible64(pos, lp, spheres, boxes):
    """Whether the segments pos -> lp (broadcast over the rows) are open."""
    t0, t1 = 1e-4, 1.0 - 1e-4
    d = lp - pos
    dd = (d * d).sum(-1)
    blocked = torch.zeros(dd.shape, dtype=torch.bool, device=DEV)
    for c in spheres:
        o = c[:3] - pos
        t = ((o * d).sum(-1) / dd).clamp(t0, t1)
        e = o - t.unsqueeze(-1) * d
        blocked |= (e * e).sum(-1) < c[3] * c[3]
    inv = 1.0 / d
    for b in boxes:
        ta, tb = (b[:3] - pos) * inv, (b[3:] - pos) * inv
        lo = torch.minimum(ta, tb).amax(-1).clamp(min=t0)
        hi = torch.maximum(ta, tb).amin(-1).clamp(max=t1)
        blocked |= lo <= hi
    return ~blocked


def _shade64(net, box, params, pos, nrm, lights):
    ws, rad = [], []
    step = max(1024, (1 << 23) // lights.shape[0])
    for p, n in zip(pos.split(step), nrm.split(step)):
        v, c = torch.sigmoid(_logits64(net, box, params, p)), _contributions64(p, n, lights)
        ws.append((v.clamp(min=0.001) * c).sum(1))
        rad.append((v * c).sum(1))
    return dict(idx=None, pdf=None, wsum=torch.cat(ws), radiance=torch.cat(rad))


def _philox(c, k0, k1):
    """Philox-4x32-10 on four int64 tensors of 32-bit words."""
    m = 0xFFFFFFFF

    def mul(a, k):
        return ((a * (k >> 16) + ((a * (k & 0xFFFF)) >> 16)) >> 16) & m, (a * k) & m

    for _ in range(10):
        h0, l0 = mul(c[0], 0xD2511F53)
        h1, l1 = mul(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return c


def _words(ids, frame, tag, block, seed):
    z = torch.zeros_like(ids)
    return _philox([ids, z + frame, z, z + ((block << 4) | tag)], seed, 0)


def _train64(case, net, box, seed, key, frame):
    """Loss and updated parameters of one training step."""
    arrays = [torch.from_numpy(a).to(DEV).double() for a in _scene_arrays(case, box, seed)]
    lights, spheres, boxes = arrays
    B = net["batch_positions"]
    nw = B - B // 2
    r = _words(torch.arange(nw, device=DEV), frame, 1, 0, key)
    world = torch.stack([(x >> 8).double() * 2.0 ** -24 for x in r[:3]], 1) * box
    screen = _view(case, box, seed)[0]
    r = _words(torch.arange(B - nw, device=DEV), frame, 2, 0, key)
    pos = torch.cat([world, screen[(r[0] * screen.shape[0]) >> 32].double()])
    if case["kind"] == "clustered":
        assign = torch.from_numpy(_clusters(case, _scene_arrays(case, box, seed)[0], seed)[1]).to(DEV).long()
        order = torch.argsort(assign, stable=True)
        cnt = torch.bincount(assign, minlength=case["clusters"])
        off = torch.cumsum(cnt, 0) - cnt
        word = torch.stack([w for b in range((case["clusters"] + 3) // 4)
                            for w in _words(torch.arange(B, device=DEV), frame, 5, b, key)], 1)
        word = word[:, :case["clusters"]]
        mem = order[(off + ((word * cnt) >> 32)).clamp(max=case["lights"] - 1)]
        target = _visible64(pos[:, None, :], lights[mem][..., :3], spheres, boxes) & (cnt > 0)
    else:
        target = _visible64(pos[:, None, :], lights[None, :, :3], spheres, boxes)
    target = target.double()
    p, m, v = (x.double() for x in _parameters(net, seed))
    p.requires_grad_(True)
    z = _logits64(net, box, p, pos)
    if net["loss"] == "bce":
        loss = torch.nn.functional.binary_cross_entropy_with_logits(z, target)
    else:
        loss = ((torch.sigmoid(z) - target) ** 2).mean()
    g, = torch.autograd.grad(loss, p)
    t, lr = STEP0 + 1, net["lr"]
    if net.get("lr_schedule") == "paper_ramp":
        lr += (net["lr_end"] - lr) * min(t - 1, net["lr_ramp_steps"]) / net["lr_ramp_steps"]
    m = BETA1 * m + (1 - BETA1) * g
    v = BETA2 * v + (1 - BETA2) * g * g
    up = m / (1 - BETA1 ** t) / ((v / (1 - BETA2 ** t)).sqrt() + EPS)
    return loss.detach(), p.detach() - lr * torch.where(m == 0, torch.zeros_like(up), up), lights


def exact(case, seed):
    net, box = _net(case)
    kind, key = case["kind"], int(seed) & 0xFFFF
    pos, nrm = _view(case, box, seed) if kind != "views" else (None, None)
    if kind in ("step", "frame", "clustered"):
        loss, p, lights = _train64(case, net, box, seed, key, 0)
        out = dict(loss=loss.reshape(1), params=p)
        if kind == "frame":
            out.update(_shade64(net, box, p, pos, nrm, lights))
        if kind == "clustered":
            vis = [torch.sigmoid(_logits64(net, box, p, x)) for x in pos.split(1 << 18)]
            out.update(vis=torch.cat(vis), light=None, weight=None, estimate=None)
        return out
    if kind == "exact_di":
        lights, spheres, boxes = (torch.from_numpy(a).to(DEV).double() for a in _scene_arrays(case, box, seed))
        out = []
        for p, n in zip(pos.split(1 << 17), nrm.split(1 << 17)):
            open_ = _visible64(p.double()[:, None, :], lights[None, :, :3], spheres, boxes)
            out.append((_contributions64(p, n, lights) * open_).sum(1))
        return torch.cat(out)
    params = _parameters(net, seed)[0].double()
    if kind == "infer":
        return torch.cat([torch.sigmoid(_logits64(net, box, params, x)) for x in pos.split(1 << 18)])
    lights = torch.from_numpy(_scene_arrays(case, box, seed)[0]).to(DEV).double()
    if kind == "views":
        return [_shade64(net, box, params, p, n, lights) for p, n in _views_of(case, box, seed)]
    out = _shade64(net, box, params, pos, nrm, lights)
    if kind == "restir":
        return dict(idx=None, pdf=None, wsum=out["wsum"], light=None, W=None, M=None, estimate=None)
    return out
