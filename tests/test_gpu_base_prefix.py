"""Base-frame spheres some of which clear the obstacles: the tests leave out the
leading clear ones only. Labels at every lane count, in the one-walk form and
in the form with centres in shared memory (a robot box asks for it), against
the pair test on the checker's own FP32 sphere centres."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("boxed", [False, True])
@pytest.mark.parametrize("near", [0, 3, 7, 8, 10, None])
def test_labels_with_some_base_spheres_clear(near, boxed):
    import torch

    from paper_2504_10783_gb300 import ezo
    from paper_2504_10783_gb300 import workloads as wl
    rd = wl.dh7_robot()
    base = np.flatnonzero(np.asarray(rd.sphere_frame) == 0)
    assert base.size == 11
    obs = wl.box_obstacles(3, 40, box_lo=(0.3, -0.5, 0.0), box_hi=(1.0, 0.5, 1.0)).spheres
    if near is not None:  # 5e-5 m from base sphere `near`, beside the column
        c, r = np.asarray(rd.sphere_xyz)[base[near]], np.asarray(rd.sphere_r)[base[near]]
        obs = np.vstack([obs, [c[0] - r - 0.004 - 5e-5, c[1], c[2], 0.004]])
    if boxed:  # far from everything
        rd.box_frame, rd.box_rot = np.zeros(1, np.int32), np.eye(3)[None]
        rd.box_xyz, rd.box_half = np.array([[0.0, 0.0, -50.0]]), np.full((1, 3), 0.01)
        rd.self_sb, rd.self_bb = np.zeros((0, 2), np.int32), np.zeros((0, 2), np.int32)
    robot, env = ezo.Robot(rd), ezo.Env(obs)
    assert ezo.check_static_spheres(robot, env) == (0 if near is not None and near < 8 else 8)
    N = 3001
    qd = torch.from_numpy(np.ascontiguousarray(wl.uniform_configs(9, rd, N).astype(np.float32).T)).cuda()
    cen = torch.empty((rd.n_spheres, 3, N), dtype=torch.float64, device="cuda")
    ezo.sphere_centres(robot, qd, cen)
    c = cen.permute(2, 0, 1).float()[:, torch.from_numpy(np.argsort(robot.sphere_order)).cuda()]
    r = torch.tensor(rd.sphere_r, dtype=torch.float32, device="cuda")
    o = torch.tensor(obs, dtype=torch.float32, device="cuda")
    p = torch.from_numpy(rd.self_pairs.astype(np.int64)).cuda()
    ratio = torch.cat([((c[:, :, None] - o[:, :3]).double().square().sum(-1)
                        / (r[:, None] + o[:, 3]).double().square()).flatten(1),
                       (c[:, p[:, 0]] - c[:, p[:, 1]]).double().square().sum(-1)
                       / (r[p[:, 0]] + r[p[:, 1]]).double().square()], 1)
    hit, close = (ratio < 1).any(1).to(torch.uint8), ((ratio - 1).abs() < 1e-6).any(1)
    assert 0.05 < hit.float().mean().item() < 0.95
    for lanes in (1, 2, 4, 8):
        flags = torch.full((N,), 7, dtype=torch.uint8, device="cuda")
        ezo.check_collision(robot, env, qd, flags, lanes=lanes)
        assert not ((flags != hit) & ~close).any(), lanes
