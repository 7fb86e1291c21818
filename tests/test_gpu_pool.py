"""Calls that borrow working memory kept between calls: the same results from
several threads on streams of their own as one after the other, and again after
the last handle has given everything back."""
import gc
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _scene():
    from paper_2504_10783_gb300 import ezo
    from paper_2504_10783_gb300 import workloads as wl
    rd = wl.planar3_robot()
    return rd, ezo.Robot(rd), ezo.Env(wl.planar_disks_candidates(3, 16) + np.array([6.0, 0.0, 0.0, 0.0]))


def test_borrowed_memory_across_threads_and_handles():
    import torch

    from paper_2504_10783_gb300 import ezo
    rng = np.random.default_rng(0)
    paths = rng.uniform(-1.0, 1.0, (6, 40, 3))
    prm = [ezo.Params.make(eps=0.1, delta=0.05, n_p=300 + 700 * i, n_mix=10, n_it_max=3, seed=i) for i in range(6)]

    def job(robot, env, i, stream):
        r = ezo.inflate_segment(robot, env, paths[i][0], paths[i][0] + 0.1, prm[i], stream=stream)
        e, n = ezo.check_path(robot, env, paths[i], 0.01, stream=stream)
        return r.status, r.A, r.b, e, n

    rd, robot, env = _scene()
    want = [job(robot, env, i, None) for i in range(6)]
    got = [None] * 24

    def work(k):
        s = torch.cuda.Stream()
        for j in range(k, 24, 4):
            got[j] = job(robot, env, j % 6, s)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    del robot, env
    gc.collect()  # the last handles: the kept blocks are freed
    rd, robot, env = _scene()
    got += [job(robot, env, i, None) for i in range(6)]
    for j, g in enumerate(got):
        for a, b in zip(want[j % 6], g):
            assert np.array_equal(a, b), j


def test_every_candidate_row_has_a_claim():
    """The two-halvings bisection (96 lanes) takes one work unit per candidate
    row, 128 a tile: with most of N_p = 1000 samples colliding its units
    outnumber 32 a tile, and the claims still have room for all of them."""
    from paper_2504_10783_gb300 import ezo
    from paper_2504_10783_gb300 import workloads as wl
    robot = ezo.Robot(wl.planar3_robot())
    # disks all around the outstretched arm: nearly every configuration but
    # the segment's surroundings collides
    ang = np.linspace(0.35, 2 * np.pi - 0.35, 60)
    disks = np.concatenate([np.column_stack([R * np.cos(ang), R * np.sin(ang), 0 * ang, 0.12 + 0 * ang])
                            for R in (0.6, 1.2, 1.8, 2.4, 2.9)])
    env = ezo.Env(disks)
    prm = ezo.Params.make(eps=0.1, delta=0.05, n_p=1000, n_f=10, n_b=10, n_mix=10, n_it_max=6, seed=1)
    got = {}
    for lanes in (8, 96):
        bt = ezo.Batch(robot, [env], np.zeros(3), np.full(3, 0.02), prm)
        bt.set_shape(bt.shape()["sample_fill_tiles"], 2, lanes)
        for step in (0, 1, 2, 3, 4):
            bt.step(step)
        bt.sync()
        assert bt.state(0)["n_cand"] > 512  # more than four tiles of 128 rows
        got[lanes] = bt.read(0, "bits")[: bt.state(0)["n_cand"]]
        bt.reset()
        bt.run()
        got[lanes] = (got[lanes], bt.segment(0).A)
    assert all(np.array_equal(a, b) for a, b in zip(got[8], got[96]))
