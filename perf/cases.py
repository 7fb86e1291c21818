"""What is timed: the calls a planner makes to this library, over the sizes it
makes them with.

A planner labels batches of configurations (roadmap and sampling checks,
``check_collision``), checks trajectories at a fine step (``check_path``),
asks for clearances (``signed_distance``), draws walks inside a polytope
(``hit_and_run``), inflates single segments, one path or many paths
(``inflate_segment``, ``Batch``, ``inflate_batch``), and, where it uses the
learned distance, trains and evaluates it (``Surrogate``). Robots and obstacle
sets are those of ``paper_2504_10783_gb300.workloads``: the planar arm, the
7-DOF arm of 40 spheres, the 11-box arm, a 10-joint chain and the Forest's
point, among disks, sphere sets of 16 to 1024 and a table-top of boxes.

``exact`` evaluates the same definitions in 64-bit torch or numpy, written
here; the inflations have none (a round's samples are chaotic 60-step walks,
and the polytopes follow from them), nor has the trained network (Adam feeds
every rounding back into the next step's gradients).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2504_10783_gb300 import ezo
from paper_2504_10783_gb300 import workloads as wl


# ------------------------------------------------------------------- cases --
def listed():
    return [
        # a planner's local check: the points of a few candidate edges of the
        # 7-DOF arm, where the call's latency is what counts
        dict(name="check_dh7_local", kind="check", robot="dh7", obstacles=64, configs=1000),
        # the batch size the paper quotes its checker on
        dict(name="check_dh7_2e6", kind="check", robot="dh7", obstacles=64, configs=2_000_000),
        # a perceived scene: a table top and objects on it as 1024 spheres
        dict(name="check_cloud", kind="check", robot="dh7_cloud", obstacles=1024, configs=200_003),
        # a planned trajectory of the box arm re-checked at a fine step among
        # table-top boxes and voxels before it is run
        dict(name="trajectory_boxes", kind="trajectory", robot="box_arm", obstacles=160, edges=300, step=0.01),
        # clearances for a roadmap or for training labels
        dict(name="clearance_dh7", kind="clearance", robot="dh7", obstacles=64, configs=131_071),
        # uniform samples of one polytope after two rounds of planes
        dict(name="walks_dh7", kind="walks", robot="dh7", walks=10_007, planes=26, steps=60),
        # the smallest inflation: one segment of the planar arm in one call
        dict(name="segment_planar3", kind="segment", robot="planar3", obstacles=16, n_p=1000, eps=0.1, steps=30),
        # the headline: a 10-segment path of the 7-DOF arm, replanned with the
        # batch a program keeps, and read back
        dict(name="path_dh7", kind="path", robot="dh7", obstacles=64, segments=10, n_p=10_000, eps=0.05, steps=60),
        # many paths over obstacle sets of different sizes in one call
        dict(name="paths_dh7", kind="paths", robot="dh7", obstacles=1024, envs=4, paths=24, segments=12, n_p=30_000,
             eps=0.05, steps=60),
        # the learned distance: evaluation, one gradient, and a short training
        dict(name="surrogate_predict", kind="predict", robot="dh7", configs=262_221),
        dict(name="surrogate_grad", kind="grad", robot="dh7", configs=3200),
        dict(name="surrogate_train", kind="train", robot="dh7", obstacles=64, configs=131_072, epochs=2, batch=3200),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["check"] * 4 + ["trajectory", "clearance", "walks", "segment", "path", "path", "paths",
                                       "predict", "grad", "train"])
    if kind == "check":
        robot = rng.choice(["dh7", "dh7", "dh7_cloud", "planar3", "chain10", "point2", "box_arm"])
        top = {"dh7_cloud": 400_000, "chain10": 500_000, "box_arm": 100_000}.get(robot, 2_000_000)
        obstacles = {"dh7": _log(rng, 16, 256), "dh7_cloud": _log(rng, 256, 1024), "planar3": rng.randint(4, 64),
                     "chain10": _log(rng, 16, 128), "point2": rng.randint(5, 30), "box_arm": 160}[robot]
        return dict(kind=kind, robot=robot, obstacles=obstacles, configs=_log(rng, 1, top))
    if kind == "trajectory":
        robot = rng.choice(["dh7", "box_arm", "planar3"])
        return dict(kind=kind, robot=robot, obstacles={"dh7": _log(rng, 16, 256), "box_arm": 160, "planar3": 16}[robot],
                    edges=_log(rng, 1, 300), step=rng.choice([0.1, 0.05, 0.01]))
    if kind == "clearance":
        robot = rng.choice(["dh7", "planar3", "chain10"])
        return dict(kind=kind, robot=robot, obstacles=_log(rng, 16, 128) if robot != "planar3" else 16,
                    configs=_log(rng, 1, 131_071))
    if kind == "walks":
        return dict(kind=kind, robot=rng.choice(["dh7", "planar3", "chain10"]), walks=_log(rng, 1, 100_000),
                    planes=rng.randint(0, 40), steps=rng.choice([30, 60]))
    if kind == "segment":
        robot = rng.choice(["planar3", "dh7", "point2", "chain10"])
        return dict(kind=kind, robot=robot, obstacles={"planar3": 16, "dh7": 64, "point2": 15, "chain10": 32}[robot],
                    n_p=_log(rng, 500, 10_000), eps=rng.choice([0.1, 0.05]), steps=30)
    if kind == "path":
        robot = rng.choice(["dh7", "dh7", "planar3"])
        return dict(kind=kind, robot=robot, obstacles=_log(rng, 32, 512) if robot == "dh7" else 16,
                    segments=rng.randint(1, 12), n_p=_log(rng, 1000, 20_000), eps=rng.choice([0.1, 0.05]), steps=60)
    if kind == "paths":
        return dict(kind=kind, robot="dh7", obstacles=_log(rng, 128, 1024), envs=rng.randint(1, 4),
                    paths=rng.randint(2, 20), segments=rng.randint(1, 10), n_p=_log(rng, 1000, 30_000), eps=0.05,
                    steps=60)
    if kind == "predict":
        return dict(kind=kind, robot="dh7", configs=_log(rng, 1, 1_048_576))
    if kind == "grad":
        return dict(kind=kind, robot="dh7", configs=64 * _log(rng, 1, 128))
    return dict(kind="train", robot="dh7", obstacles=64, configs=_log(rng, 6400, 131_072), epochs=rng.randint(1, 2),
                batch=64 * _log(rng, 4, 100))


# ------------------------------------------------------------------ inputs --
def _robot(case):
    r = case["robot"]
    return {"planar3": wl.planar3_robot, "dh7": wl.dh7_robot, "dh7_cloud": wl.dh7_robot, "chain10": wl.chain_robot,
            "point2": wl.point2_robot, "box_arm": wl.box_arm_robot}[r]()


def _env(case, seed):
    r, k = case["robot"], case["obstacles"]
    if r == "planar3":
        return wl.Env("disks", wl.planar_disks_candidates(seed, k))
    if r == "dh7_cloud":
        return wl.table_cloud_obstacles(seed, k)
    if r == "point2":
        return wl.forest_obstacles(seed, k)
    if r == "box_arm":
        return wl.tabletop_box_env(seed, k)
    if r == "chain10":  # the 1.5 m chain reaches all round: obstacles farther out
        return wl.box_obstacles(seed, k, box_lo=(0.7, -0.5, 0.0), box_hi=(1.7, 0.5, 1.0))
    return wl.box_obstacles(seed, k)


def _configs(robot, seed, count):
    """Configurations uniform in the joint limits, [n, count] float32 on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    lo = torch.tensor(robot.q_lo, dtype=torch.float32, device="cuda")[:, None]
    hi = torch.tensor(robot.q_hi, dtype=torch.float32, device="cuda")[:, None]
    return lo + (hi - lo) * torch.rand((robot.n, count), generator=g, device="cuda")


def _free_path(robot, env, rng, segments, length):
    """Waypoints of a path that keeps 0.02 m clearance (in 64 bits): from a
    start near the obstacles, each step the least clear of the free candidate
    steps, as a path around obstacles is."""
    for _ in range(50):
        q = rng.uniform(robot.q_lo, robot.q_hi, size=(2048, robot.n)) * 0.8 + 0.1 * (robot.q_lo + robot.q_hi)
        sd = _distance(robot, env, torch.tensor(q, device="cuda")).cpu().numpy()
        free = np.nonzero(sd > 0.03)[0]
        if free.size == 0:
            continue
        path = [q[free[np.argmin(sd[free])]]]
        for _ in range(segments):
            d = rng.standard_normal((96, robot.n))
            d *= length / np.linalg.norm(d, axis=1, keepdims=True)
            mid, half = 0.5 * (robot.q_lo + robot.q_hi), 0.4 * (robot.q_hi - robot.q_lo)
            end = np.clip(path[-1] + d, mid - half, mid + half)
            t = np.linspace(0.0, 1.0, 26)[None, :, None]
            pts = path[-1] + t * (end - path[-1])[:, None, :]
            c = _distance(robot, env, torch.tensor(pts.reshape(-1, robot.n), device="cuda"))
            least = c.reshape(96, 26).amin(1).cpu().numpy()
            moved = np.linalg.norm(end - path[-1], axis=1) > 0.3 * length
            ok = np.nonzero((least >= 0.02) & moved)[0]
            if ok.size == 0:
                break
            path.append(end[ok[np.argmin(least[ok])]])
        if len(path) == segments + 1:
            return np.asarray(path)
    raise RuntimeError("no free path in this scene")


def _step(case):
    return 1.0 if case["robot"] == "point2" else 0.5


def _params(case, seed):
    return ezo.Params.make(eps=case["eps"], delta=0.05, n_p=case["n_p"], n_f=10, n_b=10, n_mix=case["steps"],
                           seed=seed + 1)


def _polytope(case, seed):
    """The joint box, then planes beside a segment (A, b, v1, v2)."""
    robot, rng = _robot(case), np.random.default_rng(seed)
    n, mid, half = robot.n, 0.5 * (robot.q_lo + robot.q_hi), 0.4 * (robot.q_hi - robot.q_lo)
    v1 = mid + half * rng.uniform(-1, 1, n)
    d = rng.standard_normal(n)
    v2 = np.clip(v1 + 0.5 * d / np.linalg.norm(d), mid - half, mid + half)
    a = rng.standard_normal((case["planes"], n))
    a /= np.linalg.norm(a, axis=1, keepdims=True)
    off = np.maximum(a @ v1, a @ v2) + rng.uniform(0.05, 0.6, case["planes"])
    A = np.concatenate([np.eye(n), -np.eye(n), a])
    return A, np.concatenate([robot.q_hi, -robot.q_lo, off]), v1, v2


def _network(seed):
    """Weights as a trained network has them in size: uniform by fan-in, the
    padding features without weight; flat W1 [256 x 64], b1, W2, b2, W3, b3, w4, b4."""
    rng = np.random.default_rng(seed)
    u = lambda shape, fan: rng.uniform(-1.7, 1.7, shape) / math.sqrt(fan)  # noqa: E731
    W1 = u((256, 64), 14)
    W1[:, 14:] = 0.0
    parts = [W1, u(256, 14), u((256, 256), 256), u(256, 256), u((256, 256), 256), u(256, 256), u(256, 256), u(1, 256)]
    return np.concatenate([p.reshape(-1) for p in parts]).astype(np.float32)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("predict", "grad"):
        rd = _robot(case)
        robot = ezo.Robot(rd)
        sur = ezo.Surrogate(robot, seed=1)
        sur.set_params(_network(seed))
        q = _configs(rd, seed, case["configs"])
        state = dict(kind=kind, sur=sur, q=q)
        if kind == "predict":
            state["out"] = torch.empty(case["configs"], dtype=torch.float32, device="cuda")
        else:
            state["t"] = _targets(case, seed)
        return state
    rd = _robot(case)
    robot = ezo.Robot(rd)
    if kind == "walks":
        A, b, v1, v2 = _polytope(case, seed)
        return dict(kind=kind, A=torch.tensor(A, device="cuda"), b=torch.tensor(b, device="cuda"), v1=v1, v2=v2,
                    walks=case["walks"], steps=case["steps"], seed=seed,
                    out=torch.empty((rd.n, case["walks"]), dtype=torch.float32, device="cuda"))
    if kind == "paths":
        rng = np.random.default_rng(seed)
        sizes = [case["obstacles"]] + [int(x) for x in rng.integers(128, case["obstacles"] + 1, case["envs"] - 1)]
        scenes = [wl.box_obstacles(1000 * seed + e, k) for e, k in enumerate(sizes)]
        which = [i % case["envs"] for i in range(case["paths"])]
        # lengths 1 to `segments`, sample counts spread over a decade below n_p
        paths = [_free_path(rd, scenes[e], rng, 1 + (7 * i) % case["segments"], 0.5)
                 for i, e in enumerate(which)]
        n_seg = sum(len(p) - 1 for p in paths)
        n_p = np.exp(rng.uniform(math.log(max(500, case["n_p"] / 10)), math.log(case["n_p"]), n_seg)).astype(np.int32)
        return dict(kind=kind, robot=robot, envs=[ezo.Env(s) for s in scenes], paths=paths, which=which, n_p=n_p,
                    prm=_params(case, seed))
    scene = _env(case, seed)
    env = ezo.Env(scene)
    if kind in ("check", "clearance"):
        out = torch.empty(case["configs"], dtype=torch.uint8 if kind == "check" else torch.float32, device="cuda")
        return dict(kind=kind, robot=robot, env=env, q=_configs(rd, seed, case["configs"]), out=out)
    if kind == "trajectory":
        verts = _waypoints(case, rd, seed)
        _, total = ezo.path_points(verts, case["step"])
        return dict(kind=kind, robot=robot, env=env, verts=verts, step=case["step"],
                    out=torch.empty(total, dtype=torch.uint8, device="cuda"))
    if kind == "train":
        return dict(kind=kind, robot=robot, env=env, seed=seed, configs=case["configs"], epochs=case["epochs"],
                    batch=case["batch"])
    rng = np.random.default_rng(seed)
    for shift in range(50):  # a scene with a free path in it
        try:
            path = _free_path(rd, scene, rng, case.get("segments", 1), _step(case))
            break
        except RuntimeError:
            scene = _env(case, seed + 7919 * (shift + 1))
            env = ezo.Env(scene)
    prm = _params(case, seed)
    if kind == "segment":
        return dict(kind=kind, robot=robot, env=env, v1=path[0], v2=path[1], prm=prm)
    bt = ezo.Batch(robot, [env], path[:-1], path[1:], prm, path_first=np.zeros(len(path) - 1, np.int32))
    bt.tune()
    return dict(kind=kind, batch=bt, v1=np.ascontiguousarray(path[:-1]), v2=np.ascontiguousarray(path[1:]))


def _waypoints(case, rd, seed):
    """A random walk in the middle of the joint box, 0.497 rad an edge."""
    rng = np.random.default_rng(seed)
    mid, half = 0.5 * (rd.q_lo + rd.q_hi), 0.4 * (rd.q_hi - rd.q_lo)
    q = [mid + half * rng.uniform(-1, 1, rd.n)]
    while len(q) <= case["edges"]:
        d = rng.standard_normal(rd.n)
        nxt = q[-1] + 0.497 * d / np.linalg.norm(d)
        if np.all(np.abs(nxt - mid) <= half):
            q.append(nxt)
    return np.asarray(q)


def _targets(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed + 17)
    return -0.1 + 0.4 * torch.rand(case["configs"], generator=g, device="cuda")


# -------------------------------------------------------------------- pass --
def _table(count, n, sets):
    """Polytopes (index, A, b) as tables over `count` segments, the rows
    zero-padded to a multiple of 128."""
    rows = np.zeros(count, dtype=np.int64)
    for g, _, b in sets:
        rows[g] = len(b)
    top = max(128, -(-int(rows.max()) // 128) * 128)
    At, bt = np.zeros((count, top, n)), np.zeros((count, top))
    for g, A, b in sets:
        At[g, : len(b)], bt[g, : len(b)] = A, b
    return dict(rows=rows, A=At, b=bt)


def run(state):
    kind = state["kind"]
    if kind == "check":
        ezo.check_collision(state["robot"], state["env"], state["q"], state["out"])
        return state["out"]
    if kind == "clearance":
        ezo.signed_distance(state["robot"], state["env"], state["q"], state["out"])
        return state["out"]
    if kind == "trajectory":
        edges, points = ezo.check_path(state["robot"], state["env"], state["verts"], state["step"], state["out"])
        return dict(edges=edges.astype(np.uint8), points=points, labels=state["out"])
    if kind == "walks":
        ezo.hit_and_run(state["A"], state["b"], state["v1"], state["v2"], state["walks"], state["steps"],
                        state["seed"], 3, 2, state["out"])
        return state["out"]
    if kind == "predict":
        state["sur"].predict(state["q"], state["out"])
        return state["out"]
    if kind == "grad":
        loss, grad = state["sur"].grad(state["q"], state["t"])
        return dict(loss=np.float32(loss), grad=grad)
    if kind == "train":
        sur = ezo.Surrogate(state["robot"], seed=state["seed"] + 1)
        losses = sur.train(state["env"], state["configs"], state["epochs"], state["batch"], data_seed=state["seed"])
        return dict(losses=losses, weights=sur.params())
    if kind == "segment":
        r = ezo.inflate_segment(state["robot"], state["env"], state["v1"], state["v2"], state["prm"])
        return dict(_table(1, r.A.shape[1], [(0, r.A, r.b)]), status=r.status, rounds=r.rounds, checks=r.checks)
    if kind == "path":
        bt = state["batch"]
        bt.reset(state["v1"], state["v2"])
        bt.run_path(sequential=False, mode=ezo.RUN_GRAPH)
        status, A, b = bt.polytopes()
        return dict(_table(len(b), bt.n, list(zip(range(len(b)), A, b))), status=status)
    sets = ezo.inflate_batch(state["robot"], state["envs"], state["paths"], state["prm"], path_env=state["which"],
                             seg_np=state["n_p"], sequential=2)
    first, got = 0, []
    for path, p in zip(state["paths"], sets):
        got += [(first + k, r) for k, r in p]
        first += len(path) - 1
    out = _table(first, state["robot"].n, [(g, r.A, r.b) for g, r in got])
    for key in ("status", "rounds", "checks"):
        out[key] = np.full(first, -1, dtype=np.int64)
        for g, r in got:
            out[key][g] = getattr(r, key)
    return out


# -------------------------------------------------------------------- work --
def _check_flops(case):
    """One configuration that has to be labelled: the chain (45 flops a
    joint), every sphere's centre (18) and its distance to one obstacle (8)
    and to one sphere of the arm (8), every box's pose (72) and one test (30)."""
    r = _robot(case)
    return 45 * r.n + 34 * r.n_spheres + 102 * r.n_boxes


def work(case):
    kind, rd = case["kind"], _robot(case)
    n = rd.n
    if kind in ("check", "clearance"):
        out = 1 if kind == "check" else 4
        return dict(bytes=case["configs"] * (4 * n + out), flops=case["configs"] * _check_flops(case))
    if kind == "trajectory":
        points = case["edges"] * (0.5 / case["step"] + 1)
        return dict(bytes=8 * n * (case["edges"] + 1) + points + case["edges"], flops=points * _check_flops(case))
    walk = lambda m: 2 * m * n + 5 * m + 6 * n  # noqa: E731  (a step: every row's rate and ratio, the move)
    if kind == "walks":
        m = 2 * n + case["planes"]
        return dict(bytes=8 * m * (n + 1) + 4 * n * case["walks"], flops=case["walks"] * case["steps"] * walk(m))
    if kind == "predict":
        return dict(bytes=case["configs"] * (4 * n + 4) + 600_000, flops=case["configs"] * 2 * (2 * n + 513) * 256)
    hidden = 2 * 256 * (3 * 256 * 2 + 2 * 2 * n)  # forward and backward products of one row
    if kind == "grad":
        return dict(bytes=case["configs"] * (4 * n + 4) + 1_200_000, flops=case["configs"] * hidden)
    if kind == "train":
        rows = case["configs"] // case["batch"] * case["batch"]
        return dict(bytes=1_800_000, flops=rows * (case["epochs"] * hidden + _check_flops(case)))
    # inflations run rounds until the test accepts: one round of every segment
    # that is inflated is the least (of a path, one segment)
    segments = {"segment": 1, "path": case.get("segments", 1), "paths": case.get("paths", 1)}[kind]
    per = case["n_p"] if kind != "paths" else 0.39 * case["n_p"]
    return dict(bytes=segments * (16 * n + 16 * n * (n + 1)),
                flops=segments * per * (case["steps"] * walk(2 * n) + _check_flops(case)))


# ------------------------------------------------------------ 64-bit values --
def _frames(robot, q):
    """Rotations [N, n + 1, 3, 3] and origins [N, n + 1, 3] of the chain (q: [N, n] float64)."""
    N = q.shape[0]
    R = torch.eye(3, dtype=torch.float64, device=q.device).expand(N, 3, 3)
    o = torch.zeros((N, 3), dtype=torch.float64, device=q.device)
    Rs, os_ = [R], [o]
    for j in range(robot.n):
        slide = bool(robot.prismatic[j])
        th = (torch.zeros_like(q[:, j]) if slide else q[:, j]) + float(robot.theta_off[j])
        d = float(robot.d[j]) + (q[:, j] if slide else torch.zeros_like(q[:, j]))
        c, s = torch.cos(th), torch.sin(th)
        x = c[:, None] * R[:, :, 0] + s[:, None] * R[:, :, 1]
        y = -s[:, None] * R[:, :, 0] + c[:, None] * R[:, :, 1]
        z = R[:, :, 2]
        o = o + float(robot.a[j]) * x + d[:, None] * z
        ca, sa = math.cos(robot.alpha[j]), math.sin(robot.alpha[j])
        R = torch.stack([x, ca * y + sa * z, -sa * y + ca * z], dim=2)
        Rs.append(R)
        os_.append(o)
    return torch.stack(Rs, 1), torch.stack(os_, 1)


def _spheres(robot, R, o):
    f = torch.tensor(robot.sphere_frame, dtype=torch.long, device=R.device)
    x = torch.tensor(robot.sphere_xyz, dtype=torch.float64, device=R.device)
    return torch.einsum("nsij,sj->nsi", R[:, f], x) + o[:, f]


def _distance(robot, env, q, chunk_pairs=20_000_000):
    """Least surface distance over the obstacle and self pairs of spheres, per configuration."""
    dev = q.device
    obs = torch.tensor(env.spheres, dtype=torch.float64, device=dev)
    r = torch.tensor(robot.sphere_r, dtype=torch.float64, device=dev)
    pairs = torch.tensor(np.asarray(robot.self_pairs), dtype=torch.long, device=dev).reshape(-1, 2)
    step = max(1, chunk_pairs // max(1, robot.n_spheres * max(len(obs), 1)))
    out = []
    for i in range(0, q.shape[0], step):
        c = _spheres(robot, *_frames(robot, q[i: i + step]))
        d2 = torch.zeros((c.shape[0], c.shape[1], len(obs)), dtype=torch.float64, device=dev)
        for k in range(3):
            d2 += (c[:, :, None, k] - obs[None, None, :, k]) ** 2
        best = (d2.sqrt_() - r[None, :, None] - obs[None, None, :, 3]).amin(2).amin(1)
        if len(pairs):
            p, s = pairs[:, 0], pairs[:, 1]
            best = torch.minimum(best, ((c[:, p] - c[:, s]).norm(dim=2) - r[p] - r[s]).amin(1))
        out.append(best)
    return torch.cat(out)


def _gap_sphere_box(c, r, bc, bR, bh):
    """Distance of spheres (c [..., 3], r) to boxes (centre, axes as columns, half extents); negative inside."""
    p = torch.einsum("...ij,...i->...j", bR, c - bc).abs() - bh
    out = p.clamp(min=0).norm(dim=-1) + p.amax(-1).clamp(max=0)
    return out - r


def _gap_box_box(ac, aR, ah, bc, bR, bh):
    """Largest separation over the 15 candidate axes (positive: disjoint),
    cross products of nearly parallel edges (squared norm below 1e-4) left out."""
    axes = [aR[..., :, k] for k in range(3)] + [bR[..., :, k] for k in range(3)]
    axes += [torch.linalg.cross(*torch.broadcast_tensors(aR[..., :, i], bR[..., :, j]), dim=-1)
             for i in range(3) for j in range(3)]
    best = None
    for k, L in enumerate(axes):
        n = L.norm(dim=-1)
        u = L / n.clamp(min=1e-30)[..., None]
        ra = (torch.einsum("...ij,...i->...j", aR, u).abs() * ah).sum(-1)
        rb = (torch.einsum("...ij,...i->...j", bR, u).abs() * bh).sum(-1)
        gap = ((bc - ac) * u).sum(-1).abs() - ra - rb
        if k >= 6:
            gap = torch.where(n * n < 1e-4, torch.full_like(gap, -1e30), gap)
        best = gap if best is None else torch.maximum(best, gap)
    return best


def _box_labels(robot, env, q):
    dev, t = q.device, lambda x: torch.tensor(np.asarray(x), dtype=torch.float64, device=q.device)  # noqa: E731
    obs, eb = t(env.spheres), t(env.boxes)
    ec, eh, eR = eb[:, :3], eb[:, 3:6], eb[:, 6:].reshape(-1, 3, 3)
    f = torch.tensor(robot.box_frame, dtype=torch.long, device=dev)
    out = []
    for i in range(0, q.shape[0], 4096):
        R, o = _frames(robot, q[i: i + 4096])
        bR = R[:, f] @ t(robot.box_rot)
        bc = torch.einsum("nbij,bj->nbi", R[:, f], t(robot.box_xyz)) + o[:, f]
        bh = t(robot.box_half)
        hit = (_gap_sphere_box(obs[:, :3], obs[:, 3], bc[:, :, None], bR[:, :, None], bh[:, None]) < 0).flatten(1).any(1)
        hit |= (_gap_box_box(bc[:, :, None], bR[:, :, None], bh[:, None], ec, eR, eh) < 0).flatten(1).any(1)
        for a, b in np.asarray(robot.self_bb).reshape(-1, 2).tolist():
            hit |= _gap_box_box(bc[:, a], bR[:, a], bh[a], bc[:, b], bR[:, b], bh[b]) < 0
        out.append(hit)
    return torch.cat(out)


def _labels(case, robot, env, q):
    hit = _box_labels(robot, env, q) if robot.n_boxes else _distance(robot, env, q) < 0
    return hit.to(torch.uint8)


_M32 = np.uint64(0xFFFFFFFF)


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 of counters (arrays or scalars of 32-bit values) under a 64-bit key."""
    c = [np.broadcast_to(np.asarray(x, dtype=np.uint64), np.shape(c0)).copy() for x in (c0, c1, c2, c3)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & _M32, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & _M32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _walks(case, seed):
    """The hit-and-run walks in 64 bits (stream 3, round 2 of the key `seed`)."""
    A, b, v1, v2 = _polytope(case, seed)
    n, N = len(v1), case["walks"]
    W = max(1, (2 * ((n + 1) // 2) + 3) // 4)
    i = np.arange(N, dtype=np.uint64)
    unit = lambda x: (x >> np.uint64(8)).astype(np.float64) * 2.0 ** -24  # noqa: E731
    x = v1 + unit(_philox(i, 0, 2, 3, seed)[0])[:, None] * (v2 - v1)
    for s in range(case["steps"]):
        w = sum((_philox(i, 1 + s * W + k, 2, 3, seed) for k in range(W)), [])
        d = np.zeros((N, n))
        for p in range((n + 1) // 2):
            rho = np.sqrt(-2.0 * np.log(unit(w[2 * p]) + 2.0 ** -24))
            ang = 2.0 * np.pi * unit(w[2 * p + 1])
            d[:, 2 * p] = rho * np.cos(ang)
            if 2 * p + 1 < n:
                d[:, 2 * p + 1] = rho * np.sin(ang)
        d /= np.maximum(np.linalg.norm(d, axis=1, keepdims=True), 1e-300)
        low = np.uint64(0xFF)
        u = ((w[0] & low) | ((w[1] & low) << np.uint64(8)) | ((w[2] & low) << np.uint64(16))).astype(np.float64) * 2.0 ** -24
        slack, rate = b - x @ A.T, d @ A.T
        with np.errstate(divide="ignore", invalid="ignore"):
            t = slack / rate
        hi = np.maximum(np.where(rate > 0, t, np.inf).min(1), 0.0)
        lo = np.minimum(np.where(rate < 0, t, -np.inf).max(1), 0.0)
        move = np.isfinite(hi) & np.isfinite(lo) & (hi - lo >= 1e-12)
        x = x + np.where(move, lo + u * (hi - lo), 0.0)[:, None] * d
    return torch.tensor(np.ascontiguousarray(x.T))


def _mlp(p, q):
    """The network on configurations q [n, N] with flat weights p, in 64 bits."""
    n = q.shape[0]
    x = torch.cat([torch.sin(q.T), torch.cos(q.T), q.new_zeros((q.shape[1], 64 - 2 * n))], 1)
    at = 0
    for rows, cols in ((256, 64), (256, 256), (256, 256)):
        Wm, at = p[at: at + rows * cols].reshape(rows, cols), at + rows * cols
        x = torch.nn.functional.silu(x @ Wm.T + p[at: at + rows])
        at += rows
    return x @ p[at: at + 256] + p[at + 256]


def exact(case, seed):
    kind, rd = case["kind"], _robot(case)
    if kind in ("segment", "path", "paths", "train"):
        return None
    if kind == "walks":
        return _walks(case, seed)
    if kind in ("predict", "grad"):
        p = torch.tensor(_network(seed), dtype=torch.float64, device="cuda", requires_grad=kind == "grad")
        q = _configs(rd, seed, case["configs"]).double()
        if kind == "predict":
            return torch.cat([_mlp(p, q[:, i: i + 65536]) for i in range(0, q.shape[1], 65536)])
        loss = ((_mlp(p, q) - _targets(case, seed).double()) ** 2).mean()
        loss.backward()
        return dict(loss=float(loss.detach()), grad=p.grad)
    env = _env(case, seed)
    if kind == "trajectory":
        v = torch.tensor(_waypoints(case, rd, seed), device="cuda")
        edges, pts = [], []
        for k in range(v.shape[0] - 1):
            e = v[k + 1] - v[k]
            pieces = max(1, math.ceil(math.sqrt(sum(float(x) ** 2 for x in e.tolist())) / case["step"]))
            pts.append(v[k] + (torch.arange(pieces + 1, dtype=torch.float64, device="cuda") / pieces)[:, None] * e)
        lab = _labels(case, rd, env, torch.cat(pts))
        at = 0
        for p in pts:
            edges.append(int(lab[at: at + len(p)].any()))
            at += len(p)
        return dict(edges=np.asarray(edges, dtype=np.uint8), points=at, labels=lab)
    q = _configs(rd, seed, case["configs"]).double().T.contiguous()
    if kind == "clearance":
        return _distance(rd, env, q)
    return _labels(case, rd, env, q)
