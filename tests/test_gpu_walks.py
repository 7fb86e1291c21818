"""Walks of a call do not depend on how many lanes share one: walk i of a
large call (one lane a walk) equals walk i of every smaller one, at the counts
where the number of lanes changes and at odd counts, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [(3, 7), (7, 40), (10, 61), (16, 33), (2, 0)])
def test_walks_of_a_prefix_are_the_same(n, m):
    import torch

    from paper_2504_10783_gb300 import ezo
    rng = np.random.default_rng(n)
    a = rng.standard_normal((max(m - 2 * n, 0), n))
    A = np.concatenate([np.eye(n), -np.eye(n), a])[:m]
    b = np.concatenate([np.full(2 * n, 2.0), 0.5 + np.abs(a).sum(1) * 0.3])[:m]
    v1, v2 = np.full(n, -0.05), np.full(n, 0.05)
    Ad, bd = torch.tensor(A, device="cuda").reshape(m, n), torch.tensor(b, device="cuda")

    def walks(N):
        out = torch.full((n, N + 3), 7.0, dtype=torch.float32, device="cuda")
        ezo.hit_and_run(Ad, bd, v1, v2, N, 13, 5, 2, 3, out)
        torch.cuda.synchronize()
        assert (out[:, N:] == 7.0).all()
        return out[:, :N]

    ref = walks(41000)
    for N in (1, 31, 10239, 10240, 24575, 24577, 40959):
        assert torch.equal(walks(N), ref[:, :N]), N
