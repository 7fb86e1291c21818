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
