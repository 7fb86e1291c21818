"""Signed distances where spheres on the fixed base frame count: nearest of
all, near one obstacle of many, touching, and with no obstacle. Within the 2e-5 m
of the other signed distance tests."""
import numpy as np
import pytest

from oracle import ezo_oracle as orc
from paper_2504_10783_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count", [1, 37, 20000])
@pytest.mark.parametrize("scene", ["nearest", "many", "touching", "none"])
def test_base_spheres_are_measured(scene, count):
    import torch

    from paper_2504_10783_gb300 import ezo
    rd = wl.dh7_robot()
    near = np.asarray([[0.13, 0.0, 0.1, 0.03], [-0.2, 0.1, 0.2, 0.05]])
    spheres = {"nearest": near, "many": np.concatenate([wl.box_obstacles(3, 300).spheres, near]),
               "touching": np.asarray([[0.11, 0.0, 0.1, 0.04]]), "none": np.zeros((0, 4))}[scene]
    env = wl.Env(scene, spheres)
    q = wl.uniform_configs(11, rd, count).astype(np.float32)
    out = torch.empty(count, device="cuda")
    ezo.signed_distance(ezo.Robot(rd), ezo.Env(env), torch.from_numpy(q.T.copy()).cuda(), out)
    n = min(count, 400)
    np.testing.assert_allclose(out.cpu().numpy()[:n], orc.signed_distance(rd, env, q[:n]), rtol=0, atol=2e-5)
