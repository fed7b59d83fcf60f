"""The calls this renderer is timed on, through its public entry points.

A case is a dict of plain values.  `kind` is the entry point a program calls:

  query    Subject.query: the field at a set of observed points
  frame    Subject.set_pose + Subject.render: a fresh pose and its image
  serve    Server.submit for several viewers' frames, then Server.wait for each
  train    Subject.train_step: forward, MSE, backward and Adam
  autograd RenderFn under torch.autograd with a loss written in torch, the pose refiner and the
           weight-volume generator trained as well
  grid     Subject.refresh_occupancy, set_pose and the posed bitfield

`shape` names the performer's network sizes, which are the repository's workloads:

  tiny     32^3 volume, 8 levels of 2^14 float32 entries, two hidden layers
  frame    64^3 volume, 16 levels of 2^19 float16 entries, three hidden layers
  sweep    tiny with 2^20 entries a level

and `field` its values: "start" (entries of +-1e-4, zero residual output: a performer before
training), "textured" (entries of +-0.5, a residual output of 0.02) and "opaque" (textured with a
density bias of 30, as a trained body stops a ray within a few samples).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2306_16541_gb300 import synth

SHAPES = {
    "tiny": dict(vol=32, levels=8, log2_t=14, n_max=256, hidden=2, half=False),
    "frame": dict(vol=64, levels=16, log2_t=19, n_max=2048, hidden=3, half=True),
    "sweep": dict(vol=32, levels=8, log2_t=20, n_max=256, hidden=2, half=False),
}
N_FRAMES, FRAME_RES = 16, 512      # training frames of one performer
REFINER = (256, 4)
CNN_CHANNELS = (1024, 512, 256, 128, 64)
TAU, DILATE, S_MIN = 0.9, 1, 1e-3
LR, BETAS, EPS = 1e-4, (0.9, 0.99), 1e-8
LR_SCALE = (0.1, 1.0, 1.0, 0.1)
LIVE = 0.18                        # share of a box's cells that a posed performer's ellipsoids cover


def _frame(name, shape, w, h, s, mlp, feat, field, occ, t_min):
    return dict(name=name, kind="frame", shape=shape, width=w, height=h, samples=s, mlp=mlp, feat=feat,
                field=field, occupancy=occ, t_min=t_min)


def listed():
    return [
        # a handful of rays' points, as a picking or collision query takes them: launch latency
        dict(name="query_points", kind="query", shape="frame", points=1500, mlp="bf16", feat="f16", field="textured"),
        # a point cloud at full accuracy, as geometry extraction takes it
        dict(name="query_cloud_f32", kind="query", shape="tiny", points=250007, mlp="f32", feat="f32",
             field="textured"),
        # the smallest workload: a thumbnail at full accuracy without skipping
        _frame("frame_tiny_f32", "tiny", 64, 64, 32, "f32", "f32", "textured", False, 0.0),
        # the benchmark's frame: 512 x 512, occupancy, early termination, bf16
        _frame("frame_512_bf16", "frame", 512, 512, 128, "bf16", "f16", "start", True, 1e-4),
        # the paper's resolution with a trained, opaque performer: rays end early
        _frame("frame_1024_f16", "frame", 1024, 1024, 128, "f16", "f16", "opaque", True, 1e-4),
        # the precision sweep's frame in its narrowest type: the whole box sampled, the largest call
        _frame("frame_1080p_fp8", "sweep", 1920, 1080, 192, "fp8", "f16", "textured", False, 0.0),
        # an odd viewport at full accuracy on the tensor cores
        _frame("frame_odd_f32tc", "tiny", 333, 251, 100, "f32_tc", "f32", "textured", True, 0.0),
        # a burst of viewers' requests over two resident performers through the server
        dict(name="serve_burst_bf16", kind="serve", shape="frame", requests=6, mlp="bf16", feat="f16", field="start"),
        # the paper's iteration: 6 patches of 20 x 20 rays from one image, 128 samples
        dict(name="train_patch", kind="train", shape="tiny", rays=2400, samples=128, layout="patch", field="textured"),
        # the benchmark's training step: 2^18 uniform rays
        dict(name="train_rays", kind="train", shape="tiny", rays=1 << 18, samples=128, layout="uniform",
             field="textured"),
        # the whole motion model of the paper trained with a loss of the user's own
        dict(name="autograd_full", kind="autograd", shape="tiny", rays=4800, samples=128, layout="patch",
             field="textured"),
        # occupancy refreshed from the field's density and posed, as training and serving do now and then
        dict(name="grid_refresh", kind="grid", shape="frame", grid=128, field="textured"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["query", "query", "frame", "frame", "frame", "frame", "serve", "train", "train", "autograd", "grid"])
    field = rng.choice(["start", "textured", "opaque"])
    if kind == "query":
        mlp = rng.choice(["f32", "f32_tc", "bf16", "f16", "fp8"])
        return dict(kind=kind, shape=rng.choice(["tiny", "frame"]), points=_log(rng, 1000, 1500000), mlp=mlp,
                    feat="f32" if mlp in ("f32", "f32_tc") else rng.choice(["f16", "f32"]), field=field)
    if kind == "frame":
        mlp = rng.choice(["f32", "f32_tc", "bf16", "bf16", "f16", "fp8"])
        full = mlp in ("f32", "f32_tc")
        occ = rng.random() < 0.75
        w = _log(rng, 64, 512 if full or not occ else 1280)
        h = max(48, int(w * rng.uniform(0.5, 1.0)))
        s = rng.choice([32, 64, 96, 100, 128, 192])
        return dict(kind=kind, shape=rng.choice(["tiny", "frame", "frame"]), width=w, height=h, samples=s, mlp=mlp,
                    feat="f32" if full else "f16", field=field, occupancy=occ, t_min=rng.choice([0.0, 1e-4, 1e-4]))
    if kind == "serve":
        return dict(kind=kind, shape="frame", requests=rng.randint(2, 6), mlp=rng.choice(["bf16", "f16"]), feat="f16",
                    field=field)
    if kind == "grid":
        return dict(kind=kind, shape=rng.choice(["tiny", "frame"]), grid=rng.choice([64, 128]), field="textured")
    s = rng.choice([48, 64, 96, 100, 128, 192])
    if kind == "autograd":
        return dict(kind=kind, shape="tiny", rays=_log(rng, 1200, 20000), samples=s, layout="uniform",
                    field="textured")
    return dict(kind=kind, shape=rng.choice(["tiny", "tiny", "frame"]), rays=_log(rng, 1200, 131072), samples=s,
                layout=rng.choice(["patch", "uniform"]), field=rng.choice(["start", "textured"]))


# ------------------------------------------------------------------ inputs
def _mlp_layers(rng, dims, last_std=None, zero_last=False):
    return synth.kaiming_layers(rng, dims, zero_last=zero_last, last_std=last_std)


def _performer(shape, field, seed, grid=128):
    """A performer of the given sizes in the form Subject takes; the large arrays are made on the
    GPU and handed over as the host arrays that the library reads."""
    c = SHAPES[shape]
    rngs = [np.random.default_rng(s) for s in np.random.SeedSequence(seed).spawn(4)]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    joints = synth.rest_joints(rngs[0])
    ell = synth.ellipsoids(rngs[1], joints, grid=24)
    seg = torch.from_numpy(synth.bone_segments(joints)).cuda()
    width = torch.rand(24, device="cuda", generator=gen, dtype=torch.float64) * 0.04 + 0.04
    g = torch.linspace(-1, 1, c["vol"], device="cuda", dtype=torch.float64)
    z, y, x = torch.meshgrid(g, g, g, indexing="ij")
    pts = torch.stack([x, y, z], -1).reshape(-1, 1, 3)
    a, ab = seg[None, :, 0], (seg[:, 1] - seg[:, 0])[None]
    t = (((pts - a) * ab).sum(-1) / (ab * ab).sum(-1).clamp(min=1e-12)).clamp(0, 1)
    d2 = ((pts - a - t[..., None] * ab) ** 2).sum(-1)
    logit = torch.cat([-d2 / (2 * width ** 2), torch.full_like(d2[:, :1], -3.125)], 1)
    wvol = torch.softmax(logit, 1).T.reshape(25, c["vol"], c["vol"], c["vol"]).float().cpu().numpy()
    scale = 1e-4 if field == "start" else 0.5
    table = (torch.rand(c["levels"], 1 << c["log2_t"], 2, device="cuda", generator=gen) * 2 - 1) * scale
    if c["half"] or shape == "sweep":
        table = table.half().float()
    canon = _mlp_layers(rngs[2], synth.canonical_dims(32, 64, c["hidden"]))
    res = _mlp_layers(rngs[3], synth.residual_dims(6, 64), zero_last=field == "start",
                      last_std=None if field == "start" else 0.02)
    if field == "opaque":
        canon[-1][1][3] = 30.0
    return dict(parents=synth.PARENTS.copy(), rest_joints=joints.astype(np.float32),
                box_min=np.full(3, -1, np.float32), box_max=np.full(3, 1, np.float32), wvol=wvol, wvol_res=c["vol"],
                hash_levels=c["levels"], hash_feats=2, log2_T=c["log2_t"],
                level_res=np.array(synth.level_resolutions(c["levels"], 16, c["n_max"]), np.uint32),
                hash_table=table.cpu().numpy(), mlp_in=32, mlp_width=64, mlp_hidden_layers=c["hidden"],
                mlp_layers=canon, mlp_params=synth.pack_layers(canon), res_enabled=1, res_pe_freqs=6, res_layers=res,
                res_params=synth.pack_layers(res), ellipsoids=ell, occ_grid=grid)


def _camera(rng, w, h, s):
    return synth.camera(w, h, 1.25 * h, synth.random_eye(rng), s, 0.5, 4.5, bg=(0.1, 0.2, 0.3))


def _opts(case):
    from paper_2306_16541_gb300 import nr
    tc = case["mlp"] == "f32_tc"
    return nr.make_opts("f32" if tc else case["mlp"], case["feat"], bool(case.get("occupancy")),
                        case.get("t_min", 0.0), f32_tc=tc)


def _inputs(case, seed):
    """Everything drawn from the seed, without a handle: shared by prepare() and exact()."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed + 1)
    kind = case["kind"]
    p = dict(subj=_performer(case["shape"], case["field"], seed, case.get("grid", 128)))
    if kind in ("query", "frame", "grid"):
        p["pose"] = synth.random_pose(rng)
    if kind == "query":
        # most points lie around the body, as a user's do, and some anywhere in the box
        n = case["points"]
        joints = torch.from_numpy(p["subj"]["rest_joints"]).cuda()
        pick = torch.randint(0, 24, (n,), device="cuda", generator=gen)
        x = joints[pick] + 0.08 * torch.randn(n, 3, device="cuda", generator=gen)
        box = torch.rand(n, 3, device="cuda", generator=gen) * 2 - 1
        far = torch.rand(n, 1, device="cuda", generator=gen) < 0.1
        p["x"] = torch.where(far, box, x).clamp(-0.999, 0.999).contiguous()
    elif kind == "frame":
        p["cam"] = _camera(rng, case["width"], case["height"], case["samples"])
    elif kind == "serve":
        p["subj2"] = _performer(case["shape"], case["field"], seed + 7919)
        p["reqs"] = [dict(subject=int(rng.integers(2)), pose=synth.random_pose(rng),
                          cam=_camera(rng, *[(256, 512, 512, 1024)[i % 4]] * 2, 128)) for i in range(case["requests"])]
    elif kind in ("train", "autograd"):
        poses = [synth.random_pose(rng) for _ in range(N_FRAMES)]
        p["aa"], p["rt"] = np.stack([q[0] for q in poses]), np.stack([q[1] for q in poses])
        p["cams"] = [_camera(rng, FRAME_RES, FRAME_RES, case["samples"]) for _ in range(N_FRAMES)]
        n = case["rays"]
        if case["layout"] == "patch":
            b = synth.patch_batch(seed, N_FRAMES, -(-n // 2400))
            f, px, py = (torch.from_numpy(b[k][:n].astype(np.int32)).cuda() for k in ("frame", "px", "py"))
        else:
            f = torch.randint(0, N_FRAMES, (n,), device="cuda", generator=gen, dtype=torch.int32)
            px, py = (torch.randint(0, FRAME_RES, (n,), device="cuda", generator=gen, dtype=torch.int32)
                      for _ in range(2))
        # a smooth coloured figure stands in for the captured images
        u, v = px.float() / FRAME_RES, py.float() / FRAME_RES
        ph = f.float()[:, None] * 0.7 + torch.arange(3, device="cuda")
        p["target"] = (0.5 + 0.5 * torch.sin(9 * u[:, None] + 7 * v[:, None] + ph)).contiguous()
        p["f"], p["px"], p["py"], p["step_seed"] = f, px, py, int(rng.integers(1 << 31))
    if kind == "autograd":
        p["refiner"] = synth.refiner_layers(seed + 3, *REFINER, last_std=1e-3)
        ch = list(CNN_CHANNELS) + [25]
        std = [math.sqrt(2.0 / (ch[k] * 8)) for k in range(4)] + [1e-2]
        cnn = [(torch.randn(ch[0], 256, device="cuda", generator=gen) * math.sqrt(2.0 / 256), ch[0])]
        cnn += [(torch.randn(ch[k], ch[k + 1], 4, 4, 4, device="cuda", generator=gen) * std[k], ch[k + 1])
                for k in range(5)]
        p["cnn"] = [(w.cpu().numpy(), np.zeros(n, np.float32)) for w, n in cnn]
        p["z"] = synth.cnn_latent(seed + 4)
        p["prior"] = np.log(p["subj"]["wvol"].astype(np.float64) + 1e-6).astype(np.float32)
    return p


def prepare(case, seed):
    from paper_2306_16541_gb300 import nr
    p = _inputs(case, seed)
    kind = case["kind"]
    st = dict(kind=kind, nr=nr, sub=nr.Subject(p["subj"]))
    if kind == "query":
        st["sub"].set_pose(*p["pose"])
        st.update(x=p["x"], opts=_opts(case))
    elif kind == "frame":
        st.update(pose=p["pose"], cam=nr.make_camera(p["cam"]), opts=_opts(case),
                  out=torch.empty(case["height"], case["width"], 4, device="cuda"))
    elif kind == "serve":
        subs = [st["sub"], nr.Subject(p["subj2"])]
        srv = nr.Server(max_bytes=2 * (1200 << 20), max_slots=2)
        for s in subs:
            srv.add_subject(s)
        opts = _opts(dict(case, occupancy=True, t_min=1e-4))
        outs = [torch.empty(q["cam"].height, q["cam"].width, 4, device="cuda") for q in p["reqs"]]
        st.update(srv=srv, outs=outs, reqs=[srv.request(q["subject"], q["cam"], *q["pose"], opts, o)
                                            for q, o in zip(p["reqs"], outs)])
    elif kind in ("train", "autograd"):
        st["sub"].set_frames(p["aa"], p["rt"], p["cams"])
        st.update(batch=(p["f"], p["px"], p["py"]), target=p["target"], samples=case["samples"], seed=p["step_seed"])
        if kind == "autograd":
            st["sub"].set_pose_refiner(p["refiner"])
            st["sub"].set_weight_cnn(p["cnn"], p["z"], p["prior"])
            st["params"] = st["sub"].parameters()
        else:
            st["groups"] = [st["sub"].param(g)[0] for g in st["sub"].parameter_groups()]
            for t in st["groups"]:
                t.owner = st["sub"]      # views of the performer's own buffers: they keep it alive
    elif kind == "grid":
        st["pose"] = p["pose"]
    return st


def run(st):
    nr, sub, kind = st["nr"], st["sub"], st["kind"]
    if kind == "query":
        return sub.query(st["x"], st["opts"])
    if kind == "frame":
        sub.set_pose(*st["pose"])
        return sub.render(st["cam"], st["opts"], st["out"])
    if kind == "serve":
        for i in [st["srv"].submit(r) for r in st["reqs"]]:
            st["srv"].wait(i)
        return st["outs"]
    if kind == "train":
        loss = sub.train_step(*st["batch"], st["target"], st["samples"], st["seed"], lr=LR, betas=BETAS, eps=EPS,
                              bg=(0.1, 0.2, 0.3), lr_scale=LR_SCALE)
        return [loss] + st["groups"]
    if kind == "autograd":
        for p in st["params"]:
            p.grad = None
        sub.params_changed()           # the optimiser's step before this iteration moved the weights
        rgb = nr.RenderFn.apply(sub, *st["batch"], st["samples"], st["seed"], *st["params"])
        ((rgb - st["target"]).abs().mean() + 0.2 * ((rgb - st["target"]) ** 2).mean()).backward()
        return [rgb.detach()] + [p.grad for p in st["params"]]
    sub.refresh_occupancy(TAU, DILATE, S_MIN)
    sub.set_pose(*st["pose"])
    return [a.view(np.int32) for a in (sub.canonical_occupancy(), sub.occupancy())]


# -------------------------------------------------------- what a pass needs
def _sizes(shape):
    c = SHAPES[shape]
    can = 2 * c["levels"] * 64 + 64 * 64 * (c["hidden"] - 1) + 256
    res = 39 * 64 + 2 * 64 * 64 + 103 * 64 + 192
    table = c["levels"] * (1 << c["log2_t"]) * 2
    vol = 25 * c["vol"] ** 3
    return dict(res=2 * res, can=2 * can, table=table, vol=vol, params=table + vol + can + res)


def work(case):
    z = _sizes(case["shape"])
    kind = case["kind"]
    feat = 2 if case.get("feat") == "f16" else 4
    field = z["res"] + z["can"]

    def model(n):                       # the weights that n samples can touch at most, read once
        return 4 * min(z["vol"], 192 * n) + feat * min(z["table"], 16 * z["table"] // (1 << 10) * n)

    if kind == "query":
        n = case["points"]
        return {"bytes": n * (12 + 48) + model(n), "flops": n * field}
    if kind == "frame":
        rays = case["width"] * case["height"]
        n = rays * case["samples"] * (LIVE if case["occupancy"] else 0.9)
        return {"bytes": rays * 16 + model(n), "flops": n * field}
    if kind == "serve":
        rays = sum(((256, 512, 512, 1024)[i % 4]) ** 2 for i in range(case["requests"]))
        return {"bytes": rays * 16 + 2 * model(rays), "flops": rays * 128 * LIVE * field}
    if kind == "grid":
        n = case["grid"] ** 3
        return {"bytes": 2 * n / 8 + model(n), "flops": n * (z["can"] + LIVE * z["res"])}
    n = case["rays"] * case["samples"]
    b = case["rays"] * 24 + 4 * z["params"] * (2 if kind == "autograd" else 6)
    f = 3 * n * field
    if kind == "autograd":
        ch = list(CNN_CHANNELS) + [25]
        cnn = 256 * ch[0] + 64 * sum(a * c for a, c in zip(ch[:-1], ch[1:]))
        mac = 256 * ch[0] + sum(8 * a * c * 8 ** (k + 1) for k, (a, c) in enumerate(zip(ch[:-1], ch[1:])))
        b, f = b + 8 * cnn, f + 6 * mac
    return {"bytes": b, "flops": f}


# ------------------------------------------------------- the same in 64 bits
F64 = torch.float64


def _t(a):
    return (a if isinstance(a, torch.Tensor) else torch.as_tensor(np.asarray(a))).cuda().to(F64)


def _rot(v):
    th2 = (v * v).sum(-1)
    small = th2 < 1e-12
    th = torch.sqrt(th2.clamp(min=1e-12))
    a = torch.where(small, 1 - th2 / 6, torch.sin(th) / th)[..., None, None]
    b = torch.where(small, 0.5 - th2 / 24, (1 - torch.cos(th)) / (th * th))[..., None, None]
    o = torch.zeros_like(v[..., 0])
    k = torch.stack([o, -v[..., 2], v[..., 1], v[..., 2], o, -v[..., 0], -v[..., 1], v[..., 0], o], -1)
    k = k.reshape(v.shape[:-1] + (3, 3))
    return torch.eye(3, dtype=F64, device="cuda") + a * k + b * (k @ k)


def _log_rot(r):
    a = 0.5 * torch.stack([r[..., 2, 1] - r[..., 1, 2], r[..., 0, 2] - r[..., 2, 0], r[..., 1, 0] - r[..., 0, 1]], -1)
    c = 0.5 * (r[..., 0, 0] + r[..., 1, 1] + r[..., 2, 2] - 1)
    s2 = (a * a).sum(-1)
    s = torch.sqrt(s2.clamp(min=1e-16))
    th = torch.atan2(s, c)
    return torch.where(s2 < 1e-16, 1 + th * th / 6, th / s)[..., None] * a


def _pose64(subj, aa, rt, refiner=None):
    """(R [24][3][3], t [24][3], Omega [72]): observation to canonical space per bone."""
    joints, om = _t(subj["rest_joints"]), _t(aa).reshape(24, 3)
    rot = _rot(om)
    if refiner is not None:
        h = om[1:].reshape(-1)
        for i, (w, b) in enumerate(refiner):
            h = w @ h + b
            h = torch.relu(h) if i + 1 < len(refiner) else h
        rot = torch.cat([rot[:1], _rot(h.reshape(-1, 3)) @ rot[1:]])
        om = torch.cat([om[:1], _log_rot(rot[1:])])
    world, at = [], []
    for i in range(24):
        p = int(subj["parents"][i])
        world.append(rot[i] if p < 0 else world[p] @ rot[i])
        at.append(joints[i] + _t(rt) if p < 0 else world[p] @ (joints[i] - joints[p]) + at[p])
    r = torch.stack([w.T for w in world])
    return r, joints - torch.einsum("kij,kj->ki", r, torch.stack(at)), om.reshape(-1)


def _model64(subj, grad=False):
    def leaf(a):
        return _t(a).clone().requires_grad_(grad)
    return dict(wvol=leaf(subj["wvol"]), table=leaf(subj["hash_table"]),
                mlp=[(leaf(w), leaf(b)) for w, b in subj["mlp_layers"]],
                res=[(leaf(w), leaf(b)) for w, b in subj["res_layers"]], levels=[int(n) for n in subj["level_res"]])


def _corners(i0, f):
    for k in range(8):
        o = (k & 1, (k >> 1) & 1, k >> 2)
        w = 1
        for a in range(3):
            w = w * (f[:, a] if o[a] else 1 - f[:, a])
        yield [i0[:, a] + o[a] for a in range(3)], w


def _density64(m, x):
    """(rgb, sigma, inside) of canonical points."""
    p = (x + 1) / 2
    inside = ((p >= 0) & (p <= 1)).all(1)
    p = p.clamp(0, 1)
    slots = m["table"].shape[1]
    feats = []
    for l, n in enumerate(m["levels"]):
        pos = p * n
        i0 = pos.detach().floor().clamp(max=n - 1)
        acc = 0
        for (ix, iy, iz), w in _corners(i0.long(), pos - i0):
            if (n + 1) ** 3 <= slots:
                at = ix + iy * (n + 1) + iz * (n + 1) ** 2
            else:
                at = (ix ^ (iy * 2654435761) ^ (iz * 805459861)) & (slots - 1)
            acc = acc + w[:, None] * m["table"][l][at]
        feats.append(acc)
    h = torch.cat(feats, 1) * inside[:, None]
    h = torch.nn.functional.pad(h, (0, 32 - h.shape[1]))
    for w, b in m["mlp"][:-1]:
        h = torch.relu(h @ w.T + b)
    o = h @ m["mlp"][-1][0].T + m["mlp"][-1][1]
    return torch.sigmoid(o[:, :3]), o[:, 3].clamp(min=0) + torch.log1p(torch.exp(-o[:, 3].abs())), inside


def _field64(m, pose, x):
    """Observation points through the skeleton warp, the residual MLP and the canonical field."""
    rot, t, omega = pose
    r = m["wvol"].shape[1]
    num, s = 0, 0
    for i in range(24):
        p = x @ rot[i].T + t[i]
        u = (p + 1) * (r - 1) / 2
        i0 = u.detach().floor()
        w = 0
        flat = m["wvol"][i].reshape(-1)
        for (ix, iy, iz), c in _corners(i0.long(), u - i0):
            ok = (ix >= 0) & (ix < r) & (iy >= 0) & (iy < r) & (iz >= 0) & (iz < r)
            at = (iz.clamp(0, r - 1) * r + iy.clamp(0, r - 1)) * r + ix.clamp(0, r - 1)
            w = w + torch.where(ok, c * flat[at], torch.zeros((), dtype=F64, device="cuda"))
        num, s = num + w[:, None] * p, s + w
    xs = num / s.clamp(min=1e-4)[:, None]
    g = torch.cat([xs] + [fn((2.0 ** k) * math.pi * xs) for k in range(6) for fn in (torch.sin, torch.cos)], 1)
    (w1, b1), (w2, b2), (w3, b3), (w4, b4), (w5, b5) = m["res"]
    h = torch.relu(g @ w1[:, :39].T + (w1[:, 39:] @ omega + b1))
    h = torch.relu(h @ w2.T + b2)
    h = torch.relu(h @ w3.T + b3)
    h = torch.relu(torch.cat([h, g], 1) @ w4.T + b4)
    xf = xs + h @ w5.T + b5
    return (xs, s, xf) + _density64(m, xf)


def _rays(cam, px, py, dt):
    """Origin and unit directions, in the given type with one rounding per operation."""
    R, t = (torch.as_tensor(np.asarray(v, np.float32)).to(dt).cuda() for v in (cam.R, cam.t))
    o = torch.stack([-((R[0, k] * t[0] + R[1, k] * t[1]) + R[2, k] * t[2]) for k in range(3)])
    a = ((px.to(dt) + 0.5) - float(cam.cx)) / float(cam.fx)
    b = ((py.to(dt) + 0.5) - float(cam.cy)) / float(cam.fy)
    w = [(R[0, k] * a + R[1, k] * b) + R[2, k] for k in range(3)]
    n = torch.sqrt((w[0] * w[0] + w[1] * w[1]) + w[2] * w[2])
    return o, torch.stack([v / n for v in w], 1)


def _clip(o, d, near, far):
    lo, hi = torch.full_like(d[:, 0], near), torch.full_like(d[:, 0], far)
    miss = torch.zeros_like(lo, dtype=torch.bool)
    for k in range(3):
        z = d[:, k] == 0
        miss |= z & ((o[k] < -1) | (o[k] > 1))
        ta, tb = (-1 - o[k]) / d[:, k], (1 - o[k]) / d[:, k]
        lo = torch.where(z, lo, torch.maximum(lo, torch.minimum(ta, tb)))
        hi = torch.where(z, hi, torch.minimum(hi, torch.maximum(ta, tb)))
    return lo, hi, ~miss & (lo < hi)


def _bits32(subj, aa, rt, grid):
    """The posed occupancy cells of the ellipsoids, decided in 32 bits."""
    r, t, _ = _pose64(subj, aa, rt)
    r, t = r.float(), t.float()
    h = torch.tensor(2.0, device="cuda") / grid
    dil = 0.5 * torch.sqrt((h * h + h * h) + h * h)
    c = -1 + (torch.arange(grid, device="cuda").float() + 0.5) * h
    z, y, x = (v.reshape(-1) for v in torch.meshgrid(c, c, c, indexing="ij"))
    occ = torch.zeros(grid ** 3, dtype=torch.bool, device="cuda")
    ell = torch.from_numpy(subj["ellipsoids"]).cuda()
    for i in range(24):
        q = [((r[i, k, 0] * x + r[i, k, 1] * y) + r[i, k, 2] * z) + t[i, k] - ell[i, k] for k in range(3)]
        e = ell[i, 3:12].reshape(3, 3)
        s = [((e[k, 0] * q[0] + e[k, 1] * q[1]) + e[k, 2] * q[2]) / (ell[i, 12 + k] + dil) for k in range(3)]
        occ |= ((s[0] * s[0] + s[1] * s[1]) + s[2] * s[2]) <= 1
    return occ


def _image64(subj, pose, cam, occupancy, t_min):
    m, P = _model64(subj), _pose64(subj, *pose)
    occ = _bits32(subj, *pose, 128) if occupancy else None
    S, bg = cam.n_samples, _t(cam.bg)
    n = cam.width * cam.height
    img = torch.empty(n, 4, dtype=F64, device="cuda")
    step = max(256, (1 << 22) // S)
    for r0 in range(0, n, step):
        at = torch.arange(r0, min(n, r0 + step), device="cuda")
        px, py = at % cam.width, at // cam.width
        o32, d32 = _rays(cam, px, py, torch.float32)
        lo32, hi32, hit = _clip(o32, d32, cam.t_near, cam.t_far)
        live = hit[:, None].expand(-1, S)
        if occ is not None:
            D = (hi32 - lo32) / S
            tt = lo32[:, None] + (torch.arange(S, device="cuda").float() + 0.5)[None] * D[:, None]
            h = torch.tensor(2.0, device="cuda") / 128
            c = [(((o32[k] + tt * d32[:, k:k + 1]) + 1) / h).floor().nan_to_num().clamp(0, 127).long() for k in range(3)]
            live = live & occ[(c[2] * 128 + c[1]) * 128 + c[0]]
        o, d = _rays(cam, px, py, F64)
        lo, hi, _ = _clip(o, d, cam.t_near, cam.t_far)
        D = (hi - lo) / S
        alpha = torch.zeros(len(at), S, dtype=F64, device="cuda")
        rgb = torch.zeros(len(at), S, 3, dtype=F64, device="cuda")
        ri, si = live.nonzero(as_tuple=True)
        for q0 in range(0, len(ri), 1 << 19):
            a, b = ri[q0:q0 + (1 << 19)], si[q0:q0 + (1 << 19)]
            x = o + (lo[a] + (b + 0.5) * D[a])[:, None] * d[a]
            _, s, _, col, sig, inside = _field64(m, P, x)
            alpha[a, b] = torch.where(inside, -torch.expm1(-sig * D[a]) * s.clamp(max=1), 0.0)
            rgb[a, b] = col
        T = torch.cumprod(torch.cat([torch.ones_like(alpha[:, :1]), 1 - alpha], 1), 1)
        keep = (T[:, :-1] >= t_min).to(F64)          # a ray ends after the sample that takes T below t_min
        w = T[:, :-1] * alpha * keep
        end = torch.gather(T, 1, keep.sum(1).long()[:, None])[:, 0]
        img[at] = torch.cat([(w[..., None] * rgb).sum(1) + end[:, None] * bg, 1 - end[:, None]], 1)
    return img.reshape(cam.height, cam.width, 4)


def _jitter(seed, rays, S):
    m = np.uint64
    with np.errstate(over="ignore"):
        k = rays.astype(m)[:, None] * m(S) + np.arange(S, dtype=m)[None] + m(1)
        z = m(seed) + k * m(0x9E3779B97F4A7C15)
        z = (z ^ (z >> m(30))) * m(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> m(27))) * m(0x94D049BB133111EB)
        z = z ^ (z >> m(31))
    return torch.from_numpy((z >> m(40)).astype(np.float64) * 2.0 ** -24).cuda()


def _colours64(p, case, m, wvol, refiner, sel):
    """Training colours of the rays `sel` (all of one frame): (rays hit, rgb)."""
    f = int(p["f"][sel[0]])
    cam, S = p["cams"][f], case["samples"]
    px, py = p["px"][sel], p["py"][sel]
    o32, d32 = _rays(cam, px, py, torch.float32)
    hit = _clip(o32, d32, cam.t_near, cam.t_far)[2]
    o, d = _rays(cam, px, py, F64)
    lo, hi, _ = _clip(o, d, cam.t_near, cam.t_far)
    hit &= hi > lo
    rows = sel[hit]
    if not len(rows):
        return rows, None
    lo, hi, d = lo[hit], hi[hit], d[hit]
    t = lo[:, None] + (torch.arange(S, device="cuda") + _jitter(p["step_seed"], rows.cpu().numpy(), S)) \
        * ((hi - lo) / S)[:, None]
    delta = torch.cat([t[:, 1:] - t[:, :-1], hi[:, None] - t[:, -1:]], 1)
    x = (o + t[..., None] * d[:, None]).reshape(-1, 3)
    pose = _pose64(p["subj"], p["aa"][f], p["rt"][f], refiner)
    _, s, _, col, sig, inside = _field64(dict(m, wvol=wvol), pose, x)
    a = torch.where(inside, -torch.expm1(-sig * delta.reshape(-1)) * s.clamp(max=1), 0.0).reshape(-1, S)
    T = torch.cumprod(torch.cat([torch.ones_like(a[:, :1]), 1 - a], 1), 1)
    bg = torch.tensor([0.1, 0.2, 0.3] if case["kind"] == "train" else [0.0, 0.0, 0.0], device="cuda").to(F64)
    return rows, ((T[:, :-1] * a)[..., None] * col.reshape(-1, S, 3)).sum(1) + T[:, -1:] * bg


def _packed(layers):
    return torch.cat([t.reshape(-1) for w, b in layers for t in (w, b)])


def _train64(case, seed):
    p = _inputs(case, seed)
    full = case["kind"] == "autograd"
    m = _model64(p["subj"], grad=True)
    leaves = [[m["wvol"]], [m["table"]], [t for l in m["mlp"] for t in l], [t for l in m["res"] for t in l]]
    refiner, volume = None, m["wvol"]
    if full:
        refiner, cnn = ([(_t(w).requires_grad_(), _t(b).requires_grad_()) for w, b in p[k]] for k in ("refiner", "cnn"))
        leaves[0] = [t for l in cnn for t in l]
        leaves.append([t for l in refiner for t in l])
        h = torch.nn.functional.leaky_relu(cnn[0][0] @ _t(p["z"]) + cnn[0][1], 0.2).reshape(1, -1, 1, 1, 1)
        for k, (w, b) in enumerate(cnn[1:]):
            h = torch.nn.functional.conv_transpose3d(h, w, b, stride=2, padding=1)
            h = torch.nn.functional.leaky_relu(h, 0.2) if k < 4 else h
        volume = torch.softmax(h[0] + _t(p["prior"]), 0)
    target, n = p["target"].to(F64), case["rays"]
    wleaf = volume.detach().requires_grad_()      # the chunks' gradients meet here, then go through the generator
    rgb = torch.zeros(n, 3, dtype=F64, device="cuda")
    if not full:
        rgb += torch.tensor([0.1, 0.2, 0.3], device="cuda").to(F64)
    loss = torch.zeros((), dtype=F64, device="cuda")
    step = max(64, (1 << 18) // case["samples"])
    for f in range(N_FRAMES):
        of = (p["f"] == f).nonzero()[:, 0]
        for q0 in range(0, len(of), step):
            rows, c = _colours64(p, case, m, wleaf, refiner, of[q0:q0 + step])
            if c is None:
                continue
            e = c - target[rows]
            part = ((e.abs().sum() + 0.2 * (e * e).sum()) if full else (e * e).sum()) / (3 * n)
            part.backward()
            rgb[rows] = c.detach()
    if full:
        volume.backward(wleaf.grad)
        groups = [torch.cat([t.grad.reshape(-1) for t in leaves[k]]) for k in range(5)]
        return [rgb.float().to(F64)] + groups
    e = rgb - target
    loss = (e * e).sum() / (3 * n)
    m["wvol"].grad = wleaf.grad
    out = [float(loss)]
    for ts, scale in zip(leaves, LR_SCALE):
        x, g = (torch.cat([v.reshape(-1) for v in vs]) for vs in ([t.detach() for t in ts], [t.grad for t in ts]))
        out.append(x - LR * scale * g / (g.abs() + EPS))
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("train", "autograd"):
        return _train64(case, seed) if case["rays"] * case["samples"] <= 3 << 20 else None
    if kind == "grid":                   # whole bytes
        return None
    if kind == "frame" and not case["occupancy"] and case["width"] * case["height"] * case["samples"] > 1 << 25:
        return None
    with torch.no_grad():
        p = _inputs(case, seed)
        if kind == "frame":
            return _image64(p["subj"], p["pose"], p["cam"], case["occupancy"], case["t_min"])
        if kind == "serve":
            return [_image64(p["subj2" if q["subject"] else "subj"], q["pose"], q["cam"], True, 1e-4)
                    for q in p["reqs"]]
        m, P = _model64(p["subj"]), _pose64(p["subj"], *p["pose"])
        rows = []
        for x in p["x"].split(1 << 19):
            xs, s, xf, rgb, sig, inside = _field64(m, P, x.to(F64))
            rows.append(torch.cat([xs, s[:, None], xf, inside.to(F64)[:, None], rgb, sig[:, None]], 1))
        return torch.cat(rows)
