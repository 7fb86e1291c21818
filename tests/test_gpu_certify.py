"""Candidates and test counts from the labels: a batch whose segments' flags
begin at odd places, with sample counts around a thread's sixteen, a pass of
the block and several passes. Exact."""
import numpy as np
import pytest

from paper_2504_10783_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eps", [0.5, 0.02])
def test_candidates_are_the_first_colliding_samples(eps):
    from paper_2504_10783_gb300 import ezo
    rd, env = wl.planar3_robot(), wl.Env("disks", wl.planar_disks_candidates(3, 12))
    n_p = [1, 15, 16, 17, 1000, 16383, 16384, 16385, 40001, 7]
    v1 = np.tile(wl.uniform_configs(2, rd, 1), (len(n_p), 1))
    prm = ezo.Params.make(n_p=1000, eps=eps, seed=4)
    bt = ezo.Batch(ezo.Robot(rd), [ezo.Env(env)], v1, v1 + 0.05, prm, seg_np=np.asarray(n_p, dtype=np.int32))
    for step in range(4):
        bt.step(step)
    bt.sync()
    for g in range(len(n_p)):
        st = bt.state(g)
        lab = bt.read(g, "labels")[: st["n_samples"]].astype(bool)
        assert st["count"] == lab[: st["m_test"]].sum()
        want = np.nonzero(lab)[0][: n_p[g]]
        if st["status"] == ezo.SEG_ACCEPTED:
            want = want[:0]
        assert st["n_cand"] == want.size
        np.testing.assert_array_equal(bt.read(g, "cand_idx")[: want.size], want)
