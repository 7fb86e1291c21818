"""Robots whose poses need the most shared memory (16 joints, spheres on all 17
frames and off their axes) at the lane counts the checker accepts, on both sides
of the switch to larger blocks and up to the largest sphere counts that one lane
takes: the same labels at every count."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _robot(spheres):
    from paper_2504_10783_gb300 import workloads as wl
    rd = wl.chain_robot(16, a=0.12, r=0.03)
    rng = np.random.default_rng(spheres)
    frame = np.sort(np.arange(spheres) % 17)
    rd.sphere_frame = frame.astype(np.int32)
    rd.sphere_xyz = rng.uniform(-0.06, 0.06, (spheres, 3))
    rd.sphere_r = rng.uniform(0.01, 0.04, spheres)
    rd.sphere_link = frame.astype(np.int32)
    # two links of the arm's ends (few enough for the one-walk form)
    rd.self_pairs = np.asarray([(i, j) for i in range(spheres) for j in range(spheres)
                                if frame[i] == 2 and frame[j] >= 14], dtype=np.int32)
    return rd


@pytest.mark.parametrize("spheres", [17, 48, 56, 64, 104])
def test_largest_poses_at_one_lane(spheres):
    import torch

    from paper_2504_10783_gb300 import ezo
    from paper_2504_10783_gb300 import workloads as wl
    rd = _robot(spheres)
    rng = np.random.default_rng(1)
    env = ezo.Env(np.column_stack([rng.uniform((0.3, -1.0, -0.6), (1.6, 1.0, 1.2), (8, 3)), rng.uniform(0.15, 0.3, 8)]))
    robot = ezo.Robot(rd)
    for N in (38_911, 38_912, 40_000):
        qd = torch.from_numpy(np.ascontiguousarray(wl.uniform_configs(N, rd, N).astype(np.float32).T)).cuda()
        got = []
        for lanes in (1, 2, 4, 8):
            flags = torch.full((N,), 7, dtype=torch.uint8, device="cuda")
            ezo.check_collision(robot, env, qd, flags, lanes=lanes)
            got.append(flags)
        assert 0.02 < got[0].float().mean().item() < 0.98
        assert all(torch.equal(got[0], g) for g in got[1:]), N
