"""The training step where a tile of samples is not full: its empty places take
no part, whatever the weights hold."""
import numpy as np
import pytest

from oracle import mlp as R

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _step(theta, x, t):
    from paper_2602_21911_gb300 import grprec
    dev = lambda a: torch.tensor(np.asarray(a), dtype=torch.float32, device="cuda")
    n = len(x)
    grad = torch.zeros(R.NPARAM, dtype=torch.float32, device="cuda")
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    work = torch.empty(grprec.mlp_work_floats(n), dtype=torch.float32, device="cuda")
    grprec.grp_mlp_loss_grad(dev(theta), dev(x), dev(t), grad, loss, work)
    return loss.item(), grad.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("n", [1, 31, 32, 33, 4097])
def test_saturated_unit_in_a_part_tile(n):
    """A hidden unit saturated by an infinite weight has output 1 and passes no
    gradient; a sample of zeros in its place would be 0 x infinity."""
    rng = np.random.default_rng(n)
    theta = R.init(seed=2).astype(np.float32).astype(np.float64)
    x = rng.uniform(0.5, 1.5, size=(n, 6)).astype(np.float32)
    t = rng.normal(size=n).astype(np.float32)
    unit = 5
    theta[2 * 64 + unit] = 1e30                     # the same saturation in the reference
    l_ref, g_ref = R.loss_grad(theta, x.astype(np.float64), t.astype(np.float64))
    theta[2 * 64 + unit] = np.inf
    loss, g = _step(theta, x, t)
    assert loss == pytest.approx(l_ref, rel=1e-4)
    assert np.isfinite(g).all()
    assert np.linalg.norm(g - g_ref) <= 1e-4 * np.linalg.norm(g_ref)
