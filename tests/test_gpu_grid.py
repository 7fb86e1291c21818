"""Collision labels through the obstacle grid against the pair test over every
obstacle, on the checker's own FP32 sphere centres: obstacle counts around the
grid's switches (cells of at most four ids, lists, finer cells from 257 on),
spheres larger than the grid's edge, sets that get no grid (far from the
origin for their size, a single point) and configurations that are not
numbers. Both sides evaluate the same FP32 expression, so they may differ only
where its value is within a few roundings of the radius sum (1e-6 relative)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _obstacles(kind, n, rng):
    c, r = rng.uniform((0.2, -0.6, 0.0), (1.2, 0.6, 1.0), (n, 3)), rng.uniform(0.0, 0.1, n)
    if kind == "cluster":  # smaller than the robot's spheres: most centres lie outside the grid
        c, r = rng.normal((0.6, 0.0, 0.5), 0.01, (n, 3)), rng.uniform(0.0, 0.01, n)
    elif kind == "plane":  # long candidate lists above a dense layer
        c[:, 2], r[:] = 0.3, 0.02
    elif kind == "twins":  # every obstacle several times
        c, r = c[np.arange(n) // 8 * 8], r[np.arange(n) // 8 * 8]
    elif kind == "spread":  # one far outlier makes the cells large
        c[0] = (40.0, -30.0, 20.0)
    elif kind == "far":  # coordinates too large for cells of this size
        c[:, 0] += 1.0e6
    return np.column_stack([c, r])


@pytest.mark.parametrize("kind,n", [("box", 1), ("box", 4), ("box", 5), ("box", 64), ("box", 256), ("box", 257),
                                    ("box", 4096), ("cluster", 300), ("plane", 1024), ("twins", 512),
                                    ("spread", 100), ("far", 33)])
def test_grid_labels_equal_all_pairs(kind, n):
    import torch

    from paper_2504_10783_gb300 import ezo
    from paper_2504_10783_gb300 import workloads as wl
    rng = np.random.default_rng(n)
    rd = wl.chain_robot(7, a=0.2, r=0.05)
    rd.sphere_r = np.concatenate([[0.0, 0.35], rng.uniform(0.01, 0.1, rd.n_spheres - 2)])
    rd.self_pairs = np.zeros((0, 2), np.int32)
    obs = _obstacles(kind, n, rng)
    robot, env = ezo.Robot(rd), ezo.Env(obs)
    N = 1537
    q = wl.uniform_configs(n + 1, rd, N).astype(np.float32)
    q[5, 3], q[6, 0], q[7, 6] = np.nan, np.inf, -np.inf
    qd = torch.from_numpy(np.ascontiguousarray(q.T)).cuda()
    cen = torch.empty((rd.n_spheres, 3, N), dtype=torch.float64, device="cuda")
    ezo.sphere_centres(robot, qd, cen)
    c = cen.permute(2, 0, 1).float()
    r = torch.tensor(rd.sphere_r[robot.sphere_order], dtype=torch.float32, device="cuda")
    o = torch.tensor(obs, dtype=torch.float32, device="cuda")
    hit = torch.zeros(N, dtype=torch.bool, device="cuda")
    near = torch.zeros(N, dtype=torch.bool, device="cuda")
    for j0 in range(0, n, 256):
        d = c[:, :, None, :] - o[None, None, j0: j0 + 256, :3]
        ratio = d.double().square().sum(-1) / (r[:, None] + o[j0: j0 + 256, 3]).double().square()
        hit |= (ratio < 1.0).flatten(1).any(1)
        near |= ((ratio - 1.0).abs() < 1e-6).flatten(1).any(1)
    assert int(near.sum()) <= 3
    for lanes in (1, 2, 4, 8):
        flags = torch.full((N,), 7, dtype=torch.uint8, device="cuda")
        ezo.check_collision(robot, env, qd, flags, lanes=lanes)
        torch.cuda.synchronize()
        assert not ((flags != hit.to(torch.uint8)) & ~near).any(), lanes
    if kind in ("box", "plane"):
        assert 0 < int(hit.sum()) and (n > 64 or int(hit.sum()) < N)


@pytest.mark.parametrize("layout", ["links", "one_axis_each", "general", "many_links", "same_frame", "base"])
def test_lane_walk_equals_group_form(layout):
    """Labels with self pairs at every lane count, for robots that the one-walk
    form orders differently (spheres on one axis of their frames, off the axes,
    more links than its list holds, pairs on one frame, base spheres with
    pairs), against the pair tests on the FP32 sphere centres, and the round
    kernels' labels and bisections at every lane count against one another."""
    import torch

    from paper_2504_10783_gb300 import ezo
    from paper_2504_10783_gb300 import workloads as wl
    rng = np.random.default_rng(5)
    n = 11 if layout == "many_links" else 5
    rd = wl.chain_robot(n, a=0.3, r=0.05, per_link=5)
    link = rd.sphere_frame
    if layout == "one_axis_each":
        for f in range(1, n + 1):
            m = link == f
            rd.sphere_xyz[m] = 0.0
            rd.sphere_xyz[m, f % 3] = rng.uniform(-0.25, 0.1, int(m.sum()))
    elif layout == "general":
        rd.sphere_xyz = rd.sphere_xyz + rng.normal(0.0, 0.03, rd.sphere_xyz.shape)
    elif layout == "base":
        rd.sphere_frame = rd.sphere_frame - 1  # the first link's spheres sit on the fixed base frame
        link = rd.sphere_frame
    pairs = [(i, j) for i in range(rd.n_spheres) for j in range(i + 1, rd.n_spheres) if link[j] - link[i] >= 2]
    if layout == "same_frame":
        pairs.append((0, 4))
    rd.self_pairs = np.asarray(pairs, dtype=np.int32)
    obs = np.column_stack([rng.uniform((0.3, -0.8, -0.2), (1.4, 0.8, 1.0), (40, 3)), rng.uniform(0.02, 0.08, 40)])
    robot, env = ezo.Robot(rd), ezo.Env(obs)
    N = 4099
    qd = torch.from_numpy(np.ascontiguousarray(wl.uniform_configs(3, rd, N).astype(np.float32).T)).cuda()
    cen = torch.empty((rd.n_spheres, 3, N), dtype=torch.float64, device="cuda")
    ezo.sphere_centres(robot, qd, cen)
    order = np.argsort(robot.sphere_order)
    c = cen.permute(2, 0, 1).float()[:, torch.from_numpy(order).cuda()]
    r = torch.tensor(rd.sphere_r, dtype=torch.float32, device="cuda")
    o = torch.tensor(obs, dtype=torch.float32, device="cuda")
    p = torch.from_numpy(rd.self_pairs.astype(np.int64)).cuda()
    ratio = torch.cat([((c[:, :, None] - o[:, :3]).double().square().sum(-1)
                        / (r[:, None] + o[:, 3]).double().square()).flatten(1),
                       (c[:, p[:, 0]] - c[:, p[:, 1]]).double().square().sum(-1)
                       / (r[p[:, 0]] + r[p[:, 1]]).double().square()], 1)
    hit, near = (ratio < 1).any(1).to(torch.uint8), ((ratio - 1).abs() < 1e-6).any(1)
    assert int(near.sum()) <= 3 and 0.05 < hit.float().mean().item() < 0.95
    assert (ratio[:, 40 * rd.n_spheres:] < 1).any(1).sum().item() > 20  # self collisions among them
    for lanes in (1, 2, 4, 8):
        flags = torch.full((N,), 7, dtype=torch.uint8, device="cuda")
        ezo.check_collision(robot, env, qd, flags, lanes=lanes)
        assert not ((flags != hit) & ~near).any(), lanes
    free = torch.nonzero((ratio > 1.05).all(1)).flatten()[0].item()
    v = qd[:, free].cpu().numpy().astype(np.float64)
    prm = ezo.Params.make(eps=0.2, delta=0.2, n_p=700, n_f=10, n_b=10, n_mix=10, n_it_max=2, seed=3)
    ref = None
    for lanes in (1, 2, 4, 8, 16, 32, 96):
        bt = ezo.Batch(robot, [env], v, v + 1e-3, prm)
        bt.set_shape(bt.shape()["sample_fill_tiles"], min(lanes, 8), lanes)
        bt.run()
        got = (bt.read(0, "labels"), bt.read(0, "bits"), bt.segment(0).A)
        ref = ref or got
        assert all(np.array_equal(a, b) for a, b in zip(ref, got)), lanes


@pytest.mark.parametrize("kind,n", [("box", 1), ("box", 5), ("box", 64), ("box", 1023), ("cluster", 300),
                                    ("plane", 700), ("spread", 100), ("far", 33), ("none", 0)])
def test_signed_distance_equals_all_pairs(kind, n):
    """The signed distance (bounds of the obstacle grid, sphere by sphere)
    against the minimum over every pair on the checker's FP32 sphere centres:
    both round the same expression, 2e-7 of the coordinates' size apart at
    most (1e-6 m of a 1.7 m reach; of 1e6 m where the set lies that far out)."""
    import torch

    from paper_2504_10783_gb300 import ezo
    from paper_2504_10783_gb300 import workloads as wl
    rng = np.random.default_rng(n)
    rd = wl.chain_robot(7, a=0.2, r=0.05)
    rd.sphere_r = np.concatenate([[0.0, 0.35], rng.uniform(0.01, 0.1, rd.n_spheres - 2)])
    obs = _obstacles(kind, n, rng) if n else np.zeros((0, 4))
    robot, env = ezo.Robot(rd), ezo.Env(obs)
    N = 1021
    q = wl.uniform_configs(n + 1, rd, N).astype(np.float32)
    q[5, 3] = np.nan
    qd = torch.from_numpy(np.ascontiguousarray(q.T)).cuda()
    cen = torch.empty((rd.n_spheres, 3, N), dtype=torch.float64, device="cuda")
    ezo.sphere_centres(robot, qd, cen)
    c = cen.permute(2, 0, 1)[:, torch.from_numpy(np.argsort(robot.sphere_order)).cuda()]
    r = torch.tensor(rd.sphere_r, dtype=torch.float32, device="cuda").double()
    o = torch.tensor(obs, dtype=torch.float32, device="cuda").double()
    p = torch.from_numpy(rd.self_pairs.astype(np.int64)).cuda()
    ref = ((c[:, p[:, 0]] - c[:, p[:, 1]]).norm(dim=2) - r[p[:, 0]] - r[p[:, 1]])
    for j0 in range(0, n, 128):
        d = (c[:, :, None, :] - o[None, None, j0: j0 + 128, :3]).norm(dim=3) - r[:, None] - o[j0: j0 + 128, 3]
        ref = torch.cat([ref, d.flatten(1)], 1)
    ref = torch.where(ref.isnan(), torch.full_like(ref, 3.0e38), ref).amin(1)
    tol = 1e-6 if kind != "far" else 0.25
    for reps in (1, 17):  # small calls go by the collision grid's bounds, large ones by a grid of their own
        sd = torch.empty(N * reps, dtype=torch.float32, device="cuda")
        ezo.signed_distance(robot, env, qd.repeat(1, reps).contiguous(), sd)
        torch.cuda.synchronize()
        want = ref.repeat(reps)
        bad = ((sd.double() - want).abs() > tol) & ~((sd > 1e37) & (want > 1e37))
        assert not bad.any(), (reps, sd[bad][:5], want[bad][:5])
