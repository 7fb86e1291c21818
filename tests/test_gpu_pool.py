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
