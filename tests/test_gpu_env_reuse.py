"""Obstacle sets made and freed in turn, as a planner does for every scene it
perceives: memory handed on from one set to the next while calls on the earlier
one are still queued on another stream, from several threads, and sets of sizes
on both sides of the grid's switches. Labels and distances as with sets that
are kept."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_sets_in_turn_give_the_labels_of_kept_sets():
    import torch

    from paper_2504_10783_gb300 import ezo
    from paper_2504_10783_gb300 import workloads as wl
    rd = wl.dh7_robot()
    robot, N = ezo.Robot(rd), 20_000
    q = torch.from_numpy(np.ascontiguousarray(wl.uniform_configs(4, rd, N).astype(np.float32).T)).cuda()
    sets = [wl.box_obstacles(100 + k, k).spheres for k in (1, 4, 5, 64, 256, 257, 1000, 1024, 4096)]
    kept = [ezo.Env(s) for s in sets]
    labels = torch.full((len(sets), N), 7, dtype=torch.uint8, device="cuda")
    dist = torch.zeros((len(sets), N), device="cuda")
    for k, env in enumerate(kept):
        ezo.check_collision(robot, env, q, labels[k])
        ezo.signed_distance(robot, env, q, dist[k])
    torch.cuda.synchronize()
    del kept, env
    failed = []

    def work(w):
        stream = torch.cuda.Stream()
        order = np.random.default_rng(w).permutation(np.repeat(np.arange(len(sets)), 4))
        got_l = torch.full((order.size, N), 7, dtype=torch.uint8, device="cuda")
        got_d = torch.zeros((order.size, N), device="cuda")
        torch.cuda.synchronize()
        for i, k in enumerate(order):
            env = ezo.Env(sets[k])
            with torch.cuda.stream(stream):
                torch.cuda._sleep(1_000_000)  # the calls are still queued when the set is freed
            ezo.check_collision(robot, env, q, got_l[i], stream=stream)
            ezo.signed_distance(robot, env, q, got_d[i], stream=stream)
            del env
        torch.cuda.synchronize()
        at = torch.from_numpy(order).cuda()
        if not torch.equal(got_l, labels[at]) or (got_d - dist[at]).abs().max().item() > 1e-6:
            failed.append(w)

    work(0)
    threads = [threading.Thread(target=work, args=(w,)) for w in (1, 2, 3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
