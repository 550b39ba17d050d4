"""The calls whose speed is watched: what a user of the rasterizer has it do, through its public entry points.

A case names an entry point ("op"), a batch (E environments x A agent slots x K cameras of H x W pixels), the maps its
environments drive on and the options in use.  The listed cases are the five workloads of scenes/generate.py (one
small interactive environment up to the 65 536-agent rollout step), the paper-shaped chunk in each of its output
formats, and the remaining entry points at the size they are meant for; draw() spreads over the ranges between them.

ops: render       class + depth images of given poses (pic_render)
     step         bicycle update, class + depth images, the new state read back (pic_step, pic_get_state)
     rgb, rgb_aa  8-bit colour images, plain or antialiased (pic_render_rgb)
     step_rgb_aa  bicycle update and antialiased colour images (pic_step_rgb, pic_get_state)
     occlusion    class + depth images and the visible / unoccluded pixel counts of every road user (PIC_OPT_OCCLUSION)
     host         class + depth images from and to pinned host memory (pic_render_host)
     static       class + depth images without a scene and without allocation (pic_render_static)
"""
import math

import numpy as np
import torch

import paper_2607_26005_b200 as pic
from scenes.generate import (CLASS_CYCLIST, CLASS_GROUND, CLASS_PEDESTRIAN, CLASS_SIGNAL, CLASS_SKY, CLASS_VEHICLE, LANE_OFFSET,
                             NOMINAL_DIMS, default_palette, disk_triangles, grid_map, make_paper_rig, make_rig)

EPISODE = 100      # steps between two resets of the kinematic state (the stepping workload runs 100 steps)
NEAR = 0.5

# The maps of the workloads: grid nodes per side, block length, node jitter, curved connectors, roundabouts, view distance.
TOWNS = {
    "blocks": dict(n=3, block=200.0, jitter=0.0, arcs=False, rb=0, far=100.0),       # workload 0:    ~800 triangles
    "suburb": dict(n=5, block=150.0, jitter=10.0, arcs=False, rb=0, far=100.0),      # workload 1:  ~1 950
    "town": dict(n=8, block=100.0, jitter=10.0, arcs=True, rb=0, far=100.0),         # workloads 2, 4 and the paper's: ~5 640
    "city": dict(n=20, block=150.0, jitter=0.0, arcs=False, rb=16, far=150.0),       # workload 3: ~37 500
}

# "agents": platoons on lanes at 8-15 m headway, or spread uniformly along the roads; "some": a number of active slots
# drawn from U{1, A} per environment (the paper's chunks), else all are active; "users": cyclists and pedestrians among
# the vehicles, and traffic-light disks with a limited angular range.
_CASE = dict(op="render", town="town", maps=1, E=1, A=8, K=4, H=64, W=64, rig="ring", agents="platoons", some=False, users=False)


def _case(**kw):
    return dict(_CASE, **kw)


def listed():
    return [
        # one environment, one camera: a viewer or a unit test of a policy; launches and latency are all there is
        _case(name="viewer 1x8x1 64x64", town="blocks", A=8, K=1, agents="roads"),
        # stepping one environment interactively (debugging a policy, recording an episode)
        _case(name="step 1x64x4 64x64", op="step", A=64),
        # a training rollout on sparse traffic, every environment on its own map (workload 1)
        _case(name="rollout 256x32x4 64x64", town="suburb", maps=256, E=256, A=32, agents="roads"),
        # the headline: one step of 65 536 agents in dense platoons (workloads 2 and 4); four environments share a map
        _case(name="step 1024x64x4 64x64", op="step", maps=256, E=1024, A=64),
        # wide images of one large map shared by all environments (workload 3)
        _case(name="city 64x64x4 128x256", town="city", E=64, A=64, H=128, W=256),
        # the paper's chunk: about 2 048 egos on 31 map instances, its own rig at 96 x 54, as class + depth ...
        _case(name="paper chunk 96x54", maps=31, E=31, A=120, H=54, W=96, rig="paper", agents="roads", some=True),
        # ... as colour with all kinds of road users and signals ...
        _case(name="paper chunk rgb", op="rgb", maps=31, E=31, A=120, H=54, W=96, rig="paper", agents="roads", some=True, users=True),
        # ... and in the paper's format, antialiased colour
        _case(name="paper chunk rgb aa", op="rgb_aa", maps=31, E=31, A=120, H=54, W=96, rig="paper", agents="roads", some=True),
        # a few egos stepped at the top of the paper's resolution sweep (recording videos, evaluation)
        _case(name="step rgb aa 2x24x4 216x384", op="step_rgb_aa", maps=2, E=2, A=24, H=216, W=384, rig="paper"),
        # occlusion percentages of the road users for counterfactual probes, odd image size
        _case(name="occlusion 16x64x4 70x100", op="occlusion", maps=16, E=16, A=64, H=70, W=100),
        # a host program (no tensors on the device): poses up, images down
        _case(name="host 16x32x4 64x64", op="host", town="suburb", maps=16, E=16, A=32, agents="roads"),
        # a caller that may not allocate: small batch, small map
        _case(name="static 1x16x2 96x128", op="static", town="blocks", A=16, K=2, H=96, W=128, agents="roads"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# Most pixels and most 64 x 64 tiles of a drawn batch, by op: what costs no more than the largest listed case.
_MOST_PIXELS = dict(render=5e8, step=5e8, rgb=2e8, rgb_aa=6e7, step_rgb_aa=6e7, occlusion=3e7, host=5e7, static=4e6)
_MOST_TILES = dict(render=2.4e5, step=2.4e5, rgb=1e5, rgb_aa=2.5e4, step_rgb_aa=2.5e4, occlusion=2e4, host=1e5, static=4096)


def draw(rng):
    op = rng.choice(["render", "render", "step", "step", "rgb", "rgb_aa", "rgb_aa", "step_rgb_aa", "occlusion", "host", "static"])
    rig = rng.choice(["ring", "paper"])
    town = rng.choice(["blocks", "suburb"] if op == "static" else ["suburb", "town", "town", "city"])
    shape = rng.randrange(3)
    if shape == 0:                                  # square tiles, the training resolution
        H, W = rng.choice([(64, 64), (64, 128), (128, 128), (128, 256)])
    elif shape == 1:                                # 16:9, the paper's sweep from 32 x 18 up
        W = _log_int(rng, 32, 384)
        H = max(8, W * 9 // 16)
    else:                                           # anything
        H, W = _log_int(rng, 17, 300), _log_int(rng, 17, 300)
    if op == "static":
        E, A, K = _log_int(rng, 1, 4), _log_int(rng, 1, 32), rng.randint(1, 4)
        H, W = min(H, 160), min(W, 160)
    else:
        E, A, K = _log_int(rng, 1, 1024), _log_int(rng, 2, 128), rng.randint(1, 4)
    most = min(_MOST_PIXELS[op] / (K * H * W), _MOST_TILES[op] / (K * -(-H // 64) * -(-W // 64)))    # most agents
    E = max(1, min(E, int(most // A)))
    A = max(1, min(A, int(most // E)))
    maps = 1 if town == "city" or op == "static" else min(E, _log_int(rng, 1, 64))
    return _case(op=op, town=town, maps=maps, E=E, A=A, K=K, H=H, W=W, rig=rig, agents=rng.choice(["platoons", "roads"]),
                 some=rng.random() < 0.4, users=op != "static" and rng.random() < 0.3)


# ---- inputs ------------------------------------------------------------------------------------------------------------

def _rig(case):
    K, H, W = case["K"], case["H"], case["W"]
    if case["rig"] == "paper":
        return make_paper_rig(W, H)[:K]
    vfov = 90.0 if H == W else math.degrees(2 * math.atan(math.tan(math.radians(48.0)) * H / W))
    return make_rig([360.0 * k / K for k in range(K)], 90.0 if H == W else 96.0, vfov, W, H)


def _segments(nodes):
    return (np.concatenate([nodes[:-1, :].reshape(-1, 2), nodes[:, :-1].reshape(-1, 2)]),
            np.concatenate([nodes[1:, :].reshape(-1, 2), nodes[:, 1:].reshape(-1, 2)]))


def _on_roads(rng, nodes, n_env, A):
    """Agents of n_env environments of one map, uniform along its road centre-lines, (nearly all) at least 6 m apart, yaw along the
    road + N(0, 0.1)."""
    a, b = _segments(nodes)
    ln = np.linalg.norm(b - a, axis=1)
    pos, yaw = np.zeros((n_env, A, 2)), np.zeros((n_env, A))
    again = np.ones((n_env, A), bool)
    for _ in range(10):                                                  # the agents too close to an earlier one are placed anew
        k = int(again.sum())
        s = rng.choice(len(ln), size=k, p=ln / ln.sum())
        d = b[s] - a[s]
        pos[again] = a[s] + rng.uniform(size=(k, 1)) * d
        yaw[again] = np.arctan2(d[:, 1], d[:, 0]) + np.pi * rng.integers(0, 2, size=k) + rng.normal(0.0, 0.1, size=k)
        gap2 = sum((pos[:, :, None, c] - pos[:, None, :, c]) ** 2 for c in (0, 1))
        again = (np.tril(gap2 < 36.0, -1)).any(axis=2)
        if not again.any():
            break
    return pos, yaw


def _in_platoons(rng, nodes, n_env, A, per=8):
    """Platoons of eight on distinct lanes of a neighbourhood of (about) 3 x 3 nodes, headway U[8, 15] m, right-hand traffic."""
    n = nodes.shape[0]
    n_pl = -(-A // per)
    span = min(n, max(3, math.ceil((n_pl / 2 + 1) / 2)))                # enough lanes: 4 * span of them
    pos, yaw = np.zeros((n_env, n_pl * per, 2)), np.zeros((n_env, n_pl * per))
    for e in range(n_env):
        i0, j0 = rng.integers(0, n - span + 1, size=2)
        sub = nodes[i0:i0 + span, j0:j0 + span]
        lanes = np.concatenate([sub, sub[:, ::-1], sub.swapaxes(0, 1), sub.swapaxes(0, 1)[:, ::-1]])    # [4 span, span, 2]
        pick = rng.permutation(len(lanes))
        pts = lanes[pick[np.arange(n_pl) % len(lanes)]]                                                   # [n_pl, span, 2]
        d = np.diff(pts, axis=1)
        ln = np.linalg.norm(d, axis=2)
        cum = np.concatenate([np.zeros((n_pl, 1)), np.cumsum(ln, axis=1)], axis=1)
        rel = np.concatenate([np.zeros((n_pl, 1)), np.cumsum(rng.uniform(8.0, 15.0, size=(n_pl, per - 1)), axis=1)], axis=1)
        s = 2.0 + rng.uniform(size=(n_pl, 1)) * np.maximum(cum[:, -1:] - rel[:, -1:] - 4.0, 0.0) + rel
        i = np.clip((s[:, :, None] >= cum[:, None, :]).sum(2) - 1, 0, ln.shape[1] - 1)
        row = np.arange(n_pl)[:, None]
        t = d[row, i] / ln[row, i][..., None]
        p = pts[row, i] + t * (s - cum[row, i])[..., None] + LANE_OFFSET * np.stack([t[..., 1], -t[..., 0]], axis=-1)
        pos[e] = p.reshape(-1, 2)
        yaw[e] = (np.arctan2(t[..., 1], t[..., 0]) + rng.normal(0.0, 0.03, size=s.shape)).reshape(-1)
    return pos[:, :A], yaw[:, :A]


def _signals(rng, nodes):
    """A traffic-light disk on a 3 m pole by every junction, facing one of its roads, visible within 40 degrees."""
    tris = []
    for x, y in nodes.reshape(-1, 2)[:64]:
        h = 0.5 * np.pi * rng.integers(0, 4) + rng.normal(0.0, 0.1)
        c, s = math.cos(h), math.sin(h)
        tris.append(disk_triangles((x - 6.0 * c + 5.0 * s, y - 6.0 * s - 5.0 * c, 3.0), (c, s, 0.0), 0.15, n=12))
    return np.concatenate(tris)


def _world(case, rng):
    """Maps and agents of a case as numpy arrays."""
    town, E, A = TOWNS[case["town"]], case["E"], case["A"]
    env_map = np.arange(E) % case["maps"]
    tris, classes, limits = [], [], []
    pos, yaw = np.zeros((E, A, 2)), np.zeros((E, A))
    place = _in_platoons if case["agents"] == "platoons" else _on_roads
    for m in range(case["maps"]):
        gm = grid_map(int(rng.integers(1 << 31)), town["n"], town["block"], town["jitter"], town["arcs"], town["rb"])
        t, c, v = gm.tri_xyz, gm.tri_class, np.zeros(len(gm.tri_xyz), np.float32)
        if case["users"]:
            s = _signals(rng, gm.nodes)
            t, c = np.concatenate([t, s]), np.concatenate([c, np.full(len(s), CLASS_SIGNAL, np.uint8)])
            v = np.concatenate([v, np.full(len(s), math.cos(math.radians(40.0)), np.float32)])
        tris.append(t); classes.append(c); limits.append(v)
        of = np.flatnonzero(env_map == m)
        pos[of], yaw[of] = place(rng, gm.nodes, len(of), A)
    poses = np.concatenate([pos, ((yaw + np.pi) % (2 * np.pi) - np.pi)[..., None]], axis=2).astype(np.float32)
    dims = np.asarray(NOMINAL_DIMS) * rng.uniform(0.9, 1.1, size=(E, A, 3))
    users = None
    if case["users"]:
        users = rng.choice([CLASS_VEHICLE, CLASS_CYCLIST, CLASS_PEDESTRIAN], size=(E, A), p=[0.7, 0.15, 0.15]).astype(np.uint8)
        dims[users == CLASS_CYCLIST] *= np.array([1.8, 0.6, 1.7]) / NOMINAL_DIMS
        dims[users == CLASS_PEDESTRIAN] *= np.array([0.5, 0.6, 1.75]) / NOMINAL_DIMS
    active = np.ones((E, A), np.uint8)
    if case["some"]:
        active = (np.arange(A)[None, :] < rng.integers(1, A + 1, size=E)[:, None]).astype(np.uint8)
    counts = [len(t) for t in tris]
    return dict(tri_xyz=np.concatenate(tris), tri_class=np.concatenate(classes), offset=np.concatenate([[0], np.cumsum(counts)]).astype(np.int64),
                env_map=env_map.astype(np.int32), limits=np.concatenate(limits) if case["users"] else None, poses=poses,
                dims=dims.astype(np.float32), active=active, users=users, speed=rng.uniform(5.0, 15.0, size=(E, A, 1)).astype(np.float32))


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    w = _world(case, rng)
    E, A, K, H, W = (case[k] for k in "EAKHW")
    op, far = case["op"], TOWNS[case["town"]]["far"]
    st = {"op": op, "rig": _rig(case), "n": 0}
    dev = torch.device("cuda", 0)
    for k in ("poses", "dims", "active"):
        st[k] = torch.from_numpy(w[k]).to(dev)
    if not case["some"]:
        st["active"] = None
    shape = (E, A, K, H, W)
    if op == "static":
        st["batch"] = dict(E=E, A=A, K=K, H=H, W=W, near=NEAR, far=far, tri_xyz=torch.from_numpy(w["tri_xyz"]).to(dev), tri_class=torch.from_numpy(w["tri_class"]).to(dev))
        st["cls"], st["depth"] = torch.empty(shape, dtype=torch.uint8, device=dev), torch.empty(shape, dtype=torch.float16, device=dev)
        return st
    scene = st["scene"] = pic.Scene(E, A, K, H, W, NEAR, far, w["tri_xyz"], w["tri_class"], map_tri_offset=w["offset"], env_map_id=w["env_map"],
                                    agent_class=CLASS_VEHICLE, sky_class=CLASS_SKY, ground_class=CLASS_GROUND, tri_vis_cos=w["limits"])
    if w["users"] is not None:
        scene.set_agent_classes(torch.from_numpy(w["users"]).to(dev))
    if "rgb" in op:
        scene.set_palette(default_palette())
        st["rgb"] = torch.empty(shape + (3,), dtype=torch.uint8, device=dev)
    elif op == "host":
        # pinned host memory, as a host program that renders every step keeps it
        st["host"] = [torch.from_numpy(w[k]).pin_memory() for k in ("poses", "dims", "active")]
        st["cls"], st["depth"] = torch.empty(shape, dtype=torch.uint8).pin_memory(), torch.empty(shape, dtype=torch.float16).pin_memory()
    else:
        st["cls"], st["depth"] = scene.alloc_outputs()
    if op.startswith("step"):
        st["state0"] = torch.from_numpy(np.concatenate([w["poses"], w["speed"]], axis=2)).to(dev)
        gen = torch.Generator(device=dev).manual_seed(int(rng.integers(1 << 31)))
        steps = EPISODE if E * A <= 65536 else 20
        u = torch.rand((steps, E, A, 2), generator=gen, device=dev)
        st["actions"] = u * torch.tensor([5.0, 0.6], device=dev) - torch.tensor([3.0, 0.3], device=dev)   # accel U[-3, 2], steer U[-0.3, 0.3]
        st["state"] = torch.empty((E, A, 4), dtype=torch.float32, device=dev)
    if op == "occlusion":
        st["counts"] = torch.empty((E, A, K, A, 2), dtype=torch.int32, device=dev)
        scene.set_option(pic.OPT_OCCLUSION, st["counts"])
    torch.cuda.synchronize()
    return st


def run(st):
    op, rig = st["op"], st["rig"]
    if op == "static":
        return pic.render_static(rig=rig, poses=st["poses"], dims=st["dims"], out_class=st["cls"], out_depth=st["depth"], active=st["active"], **st["batch"])
    scene = st["scene"]
    if op.startswith("step"):
        i = st["n"] % len(st["actions"])
        st["n"] += 1
        if i == 0:                                  # a new episode
            scene.set_state(st["state0"], st["dims"], st["active"])
        if op == "step":
            out = scene.step(st["actions"][i], rig, st["cls"], st["depth"])
        else:
            out = (scene.step_rgb(st["actions"][i], rig, st["rgb"], antialias=True),)
        return tuple(out) + (scene.get_state(st["state"]),)
    if op in ("rgb", "rgb_aa"):
        return scene.render_rgb(st["poses"], st["dims"], rig, active=st["active"], out_rgb=st["rgb"], antialias=op == "rgb_aa")
    if op == "host":
        poses, dims, active = (t.numpy() for t in st["host"])
        scene.render_host(poses, dims, rig, st["cls"].numpy(), st["depth"].numpy(), active=active)
        return st["cls"], st["depth"]
    out = scene.render(st["poses"], st["dims"], rig, active=st["active"], out_class=st["cls"], out_depth=st["depth"])
    return tuple(out) + ((st["counts"],) if op == "occlusion" else ())


# ---- what a pass cannot do without -----------------------------------------------------------------------------------

_TRIANGLES = {"blocks": 792, "suburb": 1950, "town": 5640, "city": 37504}


def work(case):
    """Bytes: every pixel written once (class + depth, or RGB: 3 bytes), every map read once (36 bytes of vertices and a
    class per triangle), pose, size and activity of every agent, and per stepped agent its action and its state in, out
    and handed over.  Flops: about 100 per visible triangle, 8 per fragment and 3 per pixel, 11 per pixel of the
    workloads."""
    E, A, K, H, W = (case[k] for k in "EAKHW")
    px = E * A * K * H * W
    tris = case["maps"] * (_TRIANGLES[case["town"]] + (64 * 12 if case["users"] else 0))
    bytes_ = 3 * px + 37 * tris + 25 * E * A
    if case["op"].startswith("step"):
        bytes_ += 56 * E * A
    if case["op"] == "occlusion":
        bytes_ += 8 * E * A * K * A
    return {"bytes": bytes_, "flops": 11 * px}


def tolerance(case):
    """Class images and counts are whole numbers, depth is binary16: a pixel may go to another primitive where an edge
    or a depth gap is within float32 rounding (at most one in 10^4, and then its depth jumps); elsewhere depths agree to
    a unit of binary16.  Antialiased colours carry coverages of about 1e-4, so a channel near a half may round either way."""
    if case["op"] in ("rgb", "rgb_aa"):
        return {"rel": 1e-3, "differ": 2e-3 if case["op"] == "rgb_aa" else 1e-4}
    return {"rel": 1e-3, "max": 0.9, "differ": 2e-3 if case["op"] == "step_rgb_aa" else 1e-4}
