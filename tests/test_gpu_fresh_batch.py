"""What a batch reads back for the samples and candidates its rounds have not
reached is zero, whatever an earlier batch left in the memory it was handed."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_labels_and_bits_past_the_candidates_are_zero():
    from paper_2504_10783_gb300 import ezo
    from paper_2504_10783_gb300 import workloads as wl
    robot = ezo.Robot(wl.planar3_robot())
    ang = np.linspace(0.35, 2 * np.pi - 0.35, 60)
    disks = np.concatenate([np.column_stack([R * np.cos(ang), R * np.sin(ang), 0 * ang, 0.12 + 0 * ang])
                            for R in (0.6, 1.2, 1.8, 2.4, 2.9)])
    crowded, free = ezo.Env(disks), ezo.Env(np.array([[9.0, 9.0, 0.0, 0.1]]))
    prm = ezo.Params.make(eps=0.1, delta=0.05, n_p=1000, n_f=10, n_b=10, n_mix=10, n_it_max=6, seed=1)
    for _ in range(3):  # leaves full buffers behind, in several blocks
        bts = [ezo.Batch(robot, [crowded], np.zeros(3), np.full(3, 0.02), prm) for _ in range(3)]
        for bt in bts:
            for step in (0, 1, 2, 3, 4):
                bt.step(step)
            bt.sync()
            assert bt.state(0)["n_cand"] > 512 and bt.read(0, "bits").any()
        del bts, bt
        bts = [ezo.Batch(robot, [free], np.zeros(3), np.full(3, 0.02), prm) for _ in range(3)]
        for bt in bts:
            assert not bt.read(0, "labels").any() and not bt.read(0, "bits").any()
            for step in (0, 1, 2, 3, 4):
                bt.step(step)
            bt.sync()
            n = bt.state(0)["n_cand"]
            assert n < 500 and not bt.read(0, "bits")[n:].any()
        del bts, bt
