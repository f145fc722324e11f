"""Bulk Riemann problems: a block solves its problems in an order of its own,
so every problem's result must be what it is in any other place of the batch,
around the block sizes and with data that have no pattern (vacuum, states that
are not admissible, units beyond FP32)."""
import numpy as np
import pytest
import torch

from paper_2602_21911_gb300 import grprec

pytestmark = pytest.mark.gpu


def _solve(QL, QR, gamma):
    n = QL.shape[1]
    ps = torch.empty(n, dtype=torch.float64, device="cuda")
    it = torch.empty(n, dtype=torch.int32, device="cuda")
    st = torch.empty_like(it)
    grprec.grp_riemann_batch(QL.contiguous(), QR.contiguous(), ps, it, st, gamma=gamma)
    torch.cuda.synchronize()
    return ps, it, st


@pytest.mark.parametrize("n", [1, 31, 33, 9728, 9729, 77824, 77825])
@pytest.mark.parametrize("gamma", [1.4, 5.0 / 3.0])
def test_order_does_not_matter(n, gamma):
    rng = np.random.default_rng(n)
    W = np.exp(rng.uniform(-3.0, 3.0, (2, 3, n)))
    W[:, 1] = rng.uniform(-4.0, 4.0, (2, n))
    W[:, 2, ::7] *= -1.0                                   # not admissible
    unit = np.where(np.arange(n) % 5 == 0, 1e60, 1.0)      # beyond FP32
    Q = np.stack([W[:, 0] * unit, W[:, 0] * W[:, 1] * unit,
                  (W[:, 2] / (gamma - 1.0) + 0.5 * W[:, 0] * W[:, 1] ** 2) * unit], 1)
    Q = torch.from_numpy(Q).cuda()
    perm = torch.from_numpy(rng.permutation(n)).cuda()
    one = _solve(Q[0], Q[1], gamma)
    two = _solve(Q[0][:, perm], Q[1][:, perm], gamma)
    for a, b in zip(one, two):
        assert torch.equal(a[perm], b)
