"""Every row of a training batch is in its gradient once, and no other row: at
the rows beside the 128-row tiles and the 64-row chunks of the training kernels,
and at the batch's ends, one row's target is so far off that the gradient is that
row's but for a thousandth, after a larger batch has left rows as far off behind
the end of this one. A row that is missing, doubled or another batch's changes
every tensor by as much as its norm.

The bound against FP64 autograd on the weights as the tensor cores read them: at
most a dozen BF16 roundings lie between the configuration and a tensor of the
gradient, each below 2^-8 of the norm it applies to, and nothing averages over
one row."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = ((256, 64), (256, 256), (256, 256))
FAR = 1.0e6  # against errors below 1 of at most 2112 other rows
TOL = 12 * 2.0 ** -8


def reference(params, q, t):
    """Loss and gradient, one array a tensor, in FP64."""
    p = torch.tensor(params, dtype=torch.float64)
    at = 0
    for rows, cols in SIZES:  # the tensor cores' copies of W1, W2, W3
        p[at:at + rows * cols] = p[at:at + rows * cols].to(torch.bfloat16).double()
        at += rows * cols + rows
    p.requires_grad_(True)
    x = torch.cat([torch.sin(q.T), torch.cos(q.T), q.new_zeros(q.shape[1], 64 - 2 * q.shape[0])], 1).double().cpu()
    at, cuts = 0, []
    for rows, cols in SIZES:
        W, at = p[at:at + rows * cols].reshape(rows, cols), at + rows * cols
        x = torch.nn.functional.silu(x @ W.T + p[at:at + rows])
        cuts += [at, at + rows]
        at += rows
    y = x @ p[at:at + 256] + p[at + 256]
    loss = ((y - t.double().cpu()) ** 2).mean()
    loss.backward()
    return loss.item(), p.grad.numpy(), cuts + [at + 256]


@pytest.mark.parametrize("batch", [64, 128, 192, 320, 2112])
def test_each_row_counts_once(batch):
    from paper_2504_10783_gb300 import ezo
    from paper_2504_10783_gb300 import workloads as wl
    robot = ezo.Robot(wl.dh7_robot())
    sur = ezo.Surrogate(robot, seed=4)
    g = torch.Generator(device="cuda").manual_seed(batch)
    q = torch.rand((7, 2496), generator=g, device="cuda") * 4 - 2
    t = torch.rand(2496, generator=g, device="cuda") * 0.4 - 0.1
    behind = t.clone()
    behind[batch:] = -FAR
    for row in sorted({0, 63, 64, 127, 128, 191, batch // 2, batch - 65, batch - 1}):
        if not 0 <= row < batch:
            continue
        sur.grad(q, behind)
        tb = t[:batch].clone()
        tb[row] = FAR
        loss, got = sur.grad(q[:, :batch], tb)
        ref_loss, want, cuts = reference(sur.params(), q[:, :batch], tb)
        assert abs(loss - ref_loss) <= 1e-3 * ref_loss, row
        for a, b in zip(np.split(got.astype(np.float64), cuts), np.split(want, cuts)):
            assert np.linalg.norm(a - b) <= TOL * np.linalg.norm(b), row
