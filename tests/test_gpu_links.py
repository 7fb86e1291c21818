"""Self collisions of links whose segments are nearly parallel, where the
nearest points of the two lines are ill-determined: folded arms with thick
links that touch at one end of the overlap. Labels at every lane count against
the pair test on the checker's own FP32 sphere centres (both evaluate the same
FP32 expression, so they may differ only within 1e-6 of the radius sum), and the
path check's and a batch's labels against the same."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# sphere radius, spheres a link, sphere spacings by which the folded links are
# offset along each other, links off the axes of their frames
ARMS = [(0.4, 4, 3, False), (0.25, 3, 1, False), (0.3, 8, 2, False), (0.4, 4, 3, True), (0.02, 8, 2, False)]


def _arm(mid, r, per_link, off):
    from paper_2504_10783_gb300 import workloads as wl
    rd = wl.planar3_robot(r=r, spheres_per_link=per_link)
    rd.a = np.array([1.0, mid, 1.0])
    if off:  # both runs moved alike: the same distances, frames without an axis
        rd.sphere_xyz = rd.sphere_xyz + np.where(np.asarray(rd.sphere_frame) == 2, 0.0, 1.0)[:, None] * [0.0, 0.0, 0.1]
    return rd


@pytest.mark.parametrize("r,per_link,offset,off", ARMS)
def test_nearly_parallel_links(r, per_link, offset, off):
    import torch

    from paper_2504_10783_gb300 import ezo
    along, across = offset / per_link, 2 * r
    rd = _arm(np.hypot(along, across), r, per_link, off)
    robot, env = ezo.Robot(rd), ezo.Env(np.zeros((0, 4)))
    # links 1 and 3 folded along one another at the distance of their radii, a
    # millimetre to either side, tilted up to 2e-3 rad to either side
    N = 400_000
    rng = np.random.default_rng(7)
    fold = np.pi - np.arctan2(across, along) + rng.uniform(-1, 1, N) * 1e-3 / along
    q = np.stack([rng.uniform(-3, 3, N), fold, -fold + rng.uniform(-2e-3, 2e-3, N)], 1)
    q[::2, 1:] *= -1
    q = q.astype(np.float32)
    q[0] = (-0.0418730043, 2.32318282, -2.32424545)  # 9e-5 m deep at r = 0.4
    qd = torch.from_numpy(np.ascontiguousarray(q.T)).cuda()
    cen = torch.empty((rd.n_spheres, 3, N), dtype=torch.float64, device="cuda")
    ezo.sphere_centres(robot, qd, cen)
    c = cen.permute(2, 0, 1).float()  # planar3 lists its spheres by frame
    p = torch.from_numpy(rd.self_pairs.astype(np.int64)).cuda()
    ratio = (c[:, p[:, 0]] - c[:, p[:, 1]]).double().square().sum(-1) / (np.float32(r) + np.float32(r)) ** 2
    hit, near = (ratio < 1).any(1).to(torch.uint8), ((ratio - 1).abs() < 1e-6).any(1)
    assert 0.1 < hit.float().mean().item() < 0.9 and near.float().mean().item() < 0.1
    assert r != 0.4 or (hit[0] == 1 and not near[0])
    flags = torch.empty(N, dtype=torch.uint8, device="cuda")
    for lanes in (1, 2, 4, 8):
        flags.fill_(7)
        ezo.check_collision(robot, env, qd, flags, lanes=lanes)
        wrong = (flags != hit) & ~near
        assert not wrong.any(), (lanes, int(wrong.sum()), q[torch.nonzero(wrong)[0].item()])
    # the round kernels' labels on the same configurations
    v = np.array([0.0, 0.5, 0.5])
    n_p = 20_000
    prm = ezo.Params.make(eps=0.2, delta=0.2, n_p=n_p, n_f=1, n_b=10, n_mix=0, n_it_max=1, seed=3)
    bt = ezo.Batch(robot, [env], v, v + 1e-3, prm)
    for step in (0, 1):
        bt.step(step)
    bt.sync()
    bt.write_samples(0, q[:n_p].T)
    bt.step(2)
    bt.sync()
    wrong = (torch.from_numpy(bt.read(0, "labels")[:n_p]).cuda() != hit[:n_p]) & ~near[:n_p]
    assert not wrong.any(), int(wrong.sum())
    # and the path check's: edges of two points
    verts = q[:2001].astype(np.float64)
    pts = torch.empty(4000, dtype=torch.uint8, device="cuda")
    _, total = ezo.check_path(robot, env, verts, 100.0, pts)
    assert total == 4000
    wrong = (pts.view(2000, 2)[:, 0] != hit[:2000]) & ~near[:2000]
    assert not wrong.any(), int(wrong.sum())
