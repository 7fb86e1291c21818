"""Signed distances of sets with few pairs, which one lane a configuration
measures over all of them: the values of the FP64 oracle on both sides of every
line of that choice, and no robot slower than a larger one."""
import time

import numpy as np
import pytest

from oracle import ezo_oracle as orc
from paper_2504_10783_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _robot(name):
    return {"point2": wl.point2_robot, "planar3": wl.planar3_robot, "dh7": wl.dh7_robot, "chain10": wl.chain_robot}[name]()


# spheres x obstacles + self pairs, lines at 24, 48 and 288 pairs a joint of the
# chains compiled (3, 7, 16) and at 512 for robots of up to three spheres:
# point2 1 m, planar3 12 m + 16, dh7 40 m + 228, chain10 20 m + 112
@pytest.mark.parametrize("robot,counts", [("point2", (0, 1, 72, 73, 144, 145, 512, 513)), ("planar3", (0, 1, 4, 5, 10, 11)),
                                          ("dh7", (0, 1, 2, 3)), ("chain10", (0, 13, 14, 32, 33))])
@pytest.mark.parametrize("N", [1, 2111, 15999, 16000, 23999, 24000])
@pytest.mark.parametrize("far", [False, True])
def test_distances_on_both_sides_of_the_lines(robot, counts, N, far):
    import torch

    from paper_2504_10783_gb300 import ezo
    rd = _robot(robot)
    r = ezo.Robot(rd)
    q = wl.uniform_configs(N + far, rd, N).astype(np.float32)
    pick = np.unique(np.r_[0, N - 1, np.random.default_rng(1).integers(0, N, 200)])
    qd = torch.from_numpy(np.ascontiguousarray(q.T)).cuda()
    for k in counts:
        rng = np.random.default_rng(k)
        spheres = np.column_stack([rng.uniform(-0.8, 0.8, (k, 3)), rng.uniform(0.01, 0.1, k)])
        if far:
            spheres[:, :3] += 40.0
        sd = torch.full((N,), 7.0, device="cuda")
        ezo.signed_distance(r, ezo.Env(spheres), qd, sd)
        got = sd.cpu().numpy().astype(np.float64)[pick]
        if k == 0 and len(rd.self_pairs) == 0:
            assert (got > 1e30).all()
            continue
        want = orc.signed_distance(rd, wl.Env("s", spheres), q[pick].astype(np.float64))
        # FP32 positions up to 80 m away: 1e-6 m beside the robot, 4e-5 m there
        assert np.abs(got - want).max() <= (4e-5 if far or robot == "point2" else 2e-6), k


def test_a_smaller_robot_is_not_slower():
    """One obstacle and 131,071 configurations: the ten-joint chain's distances
    (132 pairs) take no longer than the twelve-joint chain's (204 pairs, always
    over all of them), by the fastest of ten; in groups they took 2.4 times as
    long."""
    import torch

    from paper_2504_10783_gb300 import ezo
    took = {}
    for joints in (10, 12):
        rd = wl.chain_robot(joints)
        robot, env = ezo.Robot(rd), ezo.Env(wl.box_obstacles(1, 1))
        q = torch.from_numpy(np.ascontiguousarray(wl.uniform_configs(1, rd, 131_071).T.astype(np.float32))).cuda()
        sd = torch.empty(131_071, device="cuda")
        best = 1e9
        for _ in range(10):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            ezo.signed_distance(robot, env, q, sd)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t0)
        took[joints] = best
    assert took[10] <= 1.2 * took[12], took
