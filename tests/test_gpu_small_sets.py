"""Obstacle sets that are small beside the robot's spheres (wider than the grid's
edge around the set, than the bounds' range, than anything), and sets without a
grid: labels at every lane count against the pair test on the checker's own FP32
sphere centres, equal but for values within 1e-6 of the radius sum, and the round
kernels' labels against the same."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3, 64, 300])
@pytest.mark.parametrize("extent,radii", [(0.02, (0.0, 0.08)), (0.02, (0.05, 0.3)), (0.2, (0.0, 0.12)),
                                          (0.2, (0.15, 0.4)), (0.5, (0.05, 0.2)), (0.8, (0.099, 0.101)),
                                          (2.0, (0.1, 0.7)), (1e-6, (0.0, 0.2)), (0.0, (0.0, 0.2))])
def test_small_sets_equal_all_pairs(extent, radii, n):
    import torch

    from paper_2504_10783_gb300 import ezo
    from paper_2504_10783_gb300 import workloads as wl
    rng = np.random.default_rng(n)
    rd = wl.chain_robot(6, a=0.22, r=0.05, per_link=3)
    rd.sphere_r = np.concatenate([[0.0], rng.uniform(*radii, rd.n_spheres - 1)])
    rd.self_pairs = np.zeros((0, 2), np.int32)
    c = np.array([0.45, 0.1, 0.35]) + extent * rng.uniform(-0.45, 0.45, (n, 3))
    obs = np.column_stack([c, extent * rng.uniform(0.0, 0.05, n)])
    robot, env = ezo.Robot(rd), ezo.Env(obs)
    N = 6001
    q = wl.uniform_configs(n, rd, N).astype(np.float32)
    q[5, 3], q[6, 0] = np.nan, np.inf
    qd = torch.from_numpy(np.ascontiguousarray(q.T)).cuda()
    cen = torch.empty((rd.n_spheres, 3, N), dtype=torch.float64, device="cuda")
    ezo.sphere_centres(robot, qd, cen)
    x = cen.permute(2, 0, 1).float()
    r = torch.tensor(rd.sphere_r[robot.sphere_order], dtype=torch.float32, device="cuda")
    o = torch.tensor(obs, dtype=torch.float32, device="cuda")
    hit = torch.zeros(N, dtype=torch.bool, device="cuda")
    near = torch.zeros(N, dtype=torch.bool, device="cuda")
    for j0 in range(0, n, 64):
        d = x[:, :, None, :] - o[None, None, j0: j0 + 64, :3]
        ratio = d.double().square().sum(-1) / (r[:, None] + o[j0: j0 + 64, 3]).double().square()
        hit |= (ratio < 1.0).flatten(1).any(1)
        near |= ((ratio - 1.0).abs() < 1e-6).flatten(1).any(1)
    assert int(near.sum()) <= 20 and 20 < int(hit.sum()) < N
    hit = hit.to(torch.uint8)
    for lanes in (1, 2, 4, 8):
        flags = torch.full((N,), 7, dtype=torch.uint8, device="cuda")
        ezo.check_collision(robot, env, qd, flags, lanes=lanes)
        assert not ((flags != hit) & ~near).any(), lanes
    v = np.zeros(6)
    prm = ezo.Params.make(eps=0.2, delta=0.2, n_p=N, n_f=1, n_b=10, n_mix=0, n_it_max=1, seed=3)
    bt = ezo.Batch(robot, [env], v, v + 1e-3, prm)
    for step in (0, 1):
        bt.step(step)
    bt.sync()
    bt.write_samples(0, q.T)
    bt.step(2)
    bt.sync()
    got = torch.from_numpy(bt.read(0, "labels")[:N]).cuda()
    assert not ((got != hit) & ~near).any()
