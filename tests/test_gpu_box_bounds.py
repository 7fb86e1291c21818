"""Robot boxes against obstacle spheres through the grid's bounds: rods along
each of their axes, plates, cubes and specks, turned at random, among spheres
near, far and very large, with more boxes than lanes
and with one. Labels equal the FP64 oracle's except within 5e-5 m of contact
(the band of the other box tests: FP32 kinematics, 1e-5 m for spheres, and
the axes of a box)."""
import dataclasses

import numpy as np
import pytest

from oracle import ezo_oracle as orc
from paper_2504_10783_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def turned(rng):
    q, r = np.linalg.qr(rng.standard_normal((3, 3)))
    q *= np.sign(np.diag(r))
    return q if np.linalg.det(q) > 0 else -q


@pytest.mark.parametrize("boxes", [1, 11, 29])
@pytest.mark.parametrize("scene", ["near", "sparse", "large", "one"])
@pytest.mark.parametrize("lanes", [2, 8])
def test_labels_equal_the_oracle(boxes, scene, lanes):
    import torch

    from paper_2504_10783_gb300 import ezo
    rng = np.random.default_rng(boxes)
    base = wl.dh7_robot()
    shapes = [(0.3, 0.02, 0.03), (0.02, 0.25, 0.02), (0.04, 0.03, 0.2), (0.12, 0.1, 0.005), (0.06, 0.06, 0.06),
              (1e-3, 2e-3, 1e-3)]
    half = np.asarray([shapes[i % len(shapes)] for i in range(boxes)])
    rd = dataclasses.replace(
        base, name="turned_boxes", sphere_frame=np.zeros(0, dtype=np.int32), sphere_xyz=np.zeros((0, 3)),
        sphere_r=np.zeros(0), sphere_link=np.zeros(0, dtype=np.int32), self_pairs=np.zeros((0, 2), dtype=np.int32),
        box_frame=np.sort(rng.integers(1, 8, boxes)).astype(np.int32), box_xyz=rng.uniform(-0.1, 0.1, (boxes, 3)),
        box_rot=np.stack([turned(rng) for _ in range(boxes)]), box_half=half,
        self_sb=np.zeros((0, 2), dtype=np.int32), self_bb=np.zeros((0, 2), dtype=np.int32))
    centre, radius = {
        "near": (rng.uniform((-1, -1, 0), (1, 1, 1.2), (60, 3)), rng.uniform(0.01, 0.08, 60)),
        "sparse": (rng.uniform(-3, 3, (40, 3)), rng.uniform(0.01, 0.4, 40)),
        "large": (np.asarray([[0.0, 0.0, -30.0], [4.0, 0.0, 1.0], [0.5, 0.9, 0.5]]), np.asarray([29.6, 3.2, 0.1])),
        "one": (np.asarray([[0.6, 0.2, 0.5]]), np.asarray([0.15])),
    }[scene]
    env = wl.Env(scene, np.column_stack([centre, radius]))
    q = wl.uniform_configs(7, rd, 3001).astype(np.float32)
    out = torch.empty(len(q), dtype=torch.uint8, device="cuda")
    ezo.check_collision(ezo.Robot(rd), ezo.Env(env), torch.from_numpy(q.T.copy()).cuda(), out, lanes=lanes)
    got = out.cpu().numpy().astype(bool)
    sd = orc.signed_distance(rd, env, q)
    clear = np.abs(sd) > 5e-5
    assert clear.mean() > 0.99
    np.testing.assert_array_equal(got[clear], (sd < 0)[clear])
