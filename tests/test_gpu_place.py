"""Placement by candidates held in registers and past them: the planes of a
round with one candidate, a warp's edge, one and two full passes of the block
and beyond are the oracle's greedy planes of the same end points. The rows
agree as in the round-by-round replay (the oracle forms the normal again from
the FP64 end point: 1e-6); order, count and step backs' signs are exact."""
import numpy as np
import pytest

from oracle import ezo_oracle as orc
from paper_2504_10783_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["planar3", "dh7", "chain10"])
@pytest.mark.parametrize("n_p", [1, 31, 33, 1023, 1024, 1025, 2047, 2049, 3100])
def test_planes_follow_the_greedy_order(kind, n_p):
    import torch

    from paper_2504_10783_gb300 import ezo
    rng = np.random.default_rng(5)
    if kind == "planar3":
        rd, env = wl.planar3_robot(), wl.Env("disks", wl.planar_disks_candidates(3, 12))
    elif kind == "dh7":
        rd, env = wl.dh7_robot(), wl.box_obstacles(3, 64, (-1, -1, 0.2), (1, 1, 1.2))
    else:
        rd, env = wl.chain_robot(10), wl.box_obstacles(3, 64, (-1, -1, 0.2), (1, 1, 1.2))
    robot = ezo.Robot(rd)
    scene = ezo.Env(env)
    q = torch.tensor(wl.uniform_configs(9, rd, 400).T.astype(np.float32), device="cuda").contiguous()
    hit = torch.empty(q.shape[1], dtype=torch.uint8, device="cuda")
    ezo.check_collision(robot, scene, q, hit)
    free = np.nonzero(hit.cpu().numpy() == 0)[0]
    v1 = q[:, free[rng.integers(len(free))]].cpu().numpy().astype(np.float64)
    v2 = v1 + 0.02
    prm = ezo.Params.make(n_p=n_p, n_f=12, eps=0.002, seed=3)
    bt = ezo.Batch(robot, [scene], v1, v2, prm)
    for step in range(5):
        bt.step(step)
    bt.sync()
    st = bt.state(0)
    nc, m0 = st["n_cand"], st["m"]
    assert nc == n_p  # as many collisions as places
    cst = bt.read(0, "c_star")[:, :nc].T
    idx = bt.read(0, "cand_idx")[:nc]
    bt.step(5)
    bt.sync()
    st = bt.state(0)
    pl = orc.place_hyperplanes(cst, idx, v1, v2, prm.n_f, prm.step_back_max, prm.t_col)
    H = pl.rows_a.shape[0]
    assert st["n_placed"] == H == st["m"] - m0
    np.testing.assert_array_equal(bt.read(0, "placed_idx")[:H], pl.order)
    np.testing.assert_allclose(bt.read(0, "placed_delta")[:H], pl.deltas, rtol=1e-9)
    res = bt.segment(0)
    np.testing.assert_allclose(res.A[m0:], pl.rows_a, rtol=1e-6, atol=1e-12)
    np.testing.assert_allclose(res.b[m0:], pl.rows_b, rtol=1e-6, atol=1e-12)
