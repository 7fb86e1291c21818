"""Path checks whose vertices go to the GPU through a page-locked block (up to
256 KB) and straight from the caller's array (more): the same points, labels and
edges; and a long path does not wait for a second copy of its vertices."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _path(rd, count, seed):
    rng = np.random.default_rng(seed)
    mid, half = 0.5 * (rd.q_lo + rd.q_hi), 0.4 * (rd.q_hi - rd.q_lo)
    t = np.arange(count)[:, None] * rng.uniform(0.5, 1.5, rd.n) * 4e-3
    return np.ascontiguousarray(mid + half * np.sin(t + rng.uniform(0, 6, rd.n)))


@pytest.mark.parametrize("edges", [1, 4032, 4033, 4034, 4096, 9001, 450_000, 600_000])
def test_edges_and_points_on_both_sides_of_the_limit(edges):
    """64 bytes a vertex (seven joints, an offset) and an edge's flag: 4,032
    edges are the last through the block, 450,000 take one of the pool's
    largest device blocks and 600,000 one of their own."""
    import torch

    from paper_2504_10783_gb300 import ezo
    from paper_2504_10783_gb300 import workloads as wl
    rd = wl.dh7_robot()
    robot, env = ezo.Robot(rd), ezo.Env(wl.box_obstacles(11, 64))
    verts = _path(rd, edges + 1, edges)
    counts, total = ezo.path_points(verts, 0.01)
    counts = np.asarray(counts)
    pieces = np.repeat(counts - 1, counts)
    first = np.cumsum(counts) - counts
    t = (np.arange(total) - np.repeat(first, counts)) / pieces
    at = np.repeat(np.arange(edges), counts)
    q = verts[at] + t[:, None] * (verts[at + 1] - verts[at])
    labels = torch.empty(total, dtype=torch.uint8, device="cuda")
    ezo.check_collision(robot, env, torch.from_numpy(np.ascontiguousarray(q.astype(np.float32).T)).cuda(), labels)
    got = torch.full((total,), 7, dtype=torch.uint8, device="cuda")
    flags, points = ezo.check_path(robot, env, verts, 0.01, got)
    assert points == total
    assert torch.equal(got, labels)
    hit = np.zeros(edges, dtype=bool)
    hit[at[labels.cpu().numpy() != 0]] = True
    np.testing.assert_array_equal(flags, hit)


def test_a_long_path_waits_for_one_copy():
    """1.2 million vertices: no more than twice what the host's own count of the
    points and one copy of the vertices to the GPU take (6.9 ms on a GB300, 14.1
    with a second copy into page-locked memory), by the fastest of eight."""
    import torch

    from paper_2504_10783_gb300 import ezo
    from paper_2504_10783_gb300 import workloads as wl
    rd = wl.dh7_robot()
    robot, env = ezo.Robot(rd), ezo.Env(wl.box_obstacles(11, 64))
    verts = _path(rd, 1_200_000, 1)

    def fastest(f):
        best = 1e9
        for _ in range(8):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            f()
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t0)
        return best

    host = torch.from_numpy(verts)
    device = torch.empty_like(host, device="cuda")
    copy = fastest(lambda: device.copy_(host))
    count = fastest(lambda: ezo.path_points(verts, 0.05))
    check = fastest(lambda: ezo.check_path(robot, env, verts, 0.05))
    print(f"copy {1e3 * copy:.2f} count {1e3 * count:.2f} check {1e3 * check:.2f} ms")
    assert check <= 2.0 * (copy + count)
