"""Self pairs tested one by one by groups with a lane or two for each (robots of
up to three joints), against their links' screen and against FP64: folded planar
arms at every lane count, with pair counts on both sides of the switch at eight
lanes (16 pairs) and four (8)."""
import dataclasses

import numpy as np
import pytest

from oracle import ezo_oracle as orc
from paper_2504_10783_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pairs", [0, 1, 4, 5, 7, 8, 9, 15, 16, 17, 25])
def test_labels_of_folded_arms(pairs):
    import torch

    from paper_2504_10783_gb300 import ezo
    base = wl.planar3_robot(spheres_per_link=5, r=0.12)
    assert len(base.self_pairs) == 25
    # whole rows and a rest of the 5 x 5 pairs, in a shuffled order and direction
    rng = np.random.default_rng(pairs)
    chosen = np.asarray(base.self_pairs)[:pairs].copy()
    flip = rng.random(pairs) < 0.5
    chosen[flip] = chosen[flip][:, ::-1]
    rd = dataclasses.replace(base, self_pairs=chosen[rng.permutation(pairs)])
    N = 20_000
    q = wl.uniform_configs(pairs, rd, N)
    q[: N // 2, 1] = np.pi + rng.normal(0, 0.3, N // 2)  # folded: links 1 and 3 near each other
    q[: N // 2, 2] = np.pi * rng.choice([-1, 1], N // 2) + rng.normal(0, 0.3, N // 2)
    q = q.astype(np.float32)
    qd = torch.from_numpy(np.ascontiguousarray(q.T)).cuda()
    env = wl.Env("s", np.array([[1.5, 1.5, 0.0, 0.2], [-1.0, 2.0, 0.0, 0.3]]))
    robot, envh = ezo.Robot(rd), ezo.Env(env)
    labels = []
    for lanes in (1, 2, 4, 8):
        fl = torch.full((N,), 7, dtype=torch.uint8, device="cuda")
        ezo.check_collision(robot, envh, qd, fl, lanes)
        labels.append(fl.cpu().numpy())
    for other in labels[1:]:
        np.testing.assert_array_equal(labels[0], other)
    sd = orc.signed_distance(rd, env, q.astype(np.float64))
    sure = np.abs(sd) >= 1e-5
    np.testing.assert_array_equal(labels[0][sure] != 0, sd[sure] < 0)
    assert 0 < labels[0].sum() < N
