"""The predictor's kernels on both sides of the batch sizes where a thread per
sample takes over from a thread per sample and hidden unit."""
import numpy as np
import pytest

from helpers import ensure_lib
from oracle import mlp

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    ensure_lib()


def _inputs(B):
    rng = np.random.default_rng(B)
    f = lambda scale, *shape: torch.from_numpy(rng.normal(0, scale, shape).astype(np.float32)).cuda()  # noqa: E731
    return f(0.25, mlp.NPARAMS), f(1, B, 8), f(1, B, 2)


@pytest.mark.parametrize("B", [8192, 8193, 32768, 32769, 40001])
def test_rows_do_not_depend_on_the_batch(B):
    """A sample's outputs and activations have the same bits in a batch of any size."""
    from paper_2010_12117_gb300 import binding
    p, x, _ = _inputs(B)
    y, ya = (torch.empty(B, 2, device="cuda") for _ in range(2))
    act = torch.empty(B, 128, device="cuda")
    binding.mlp_forward(p, x, y)
    binding.mlp_forward(p, x, ya, act)
    part, pact = torch.empty_like(y), torch.empty_like(act)
    for lo in range(0, B, 1000):
        hi = min(B, lo + 1000)
        binding.mlp_forward(p, x[lo:hi], part[lo:hi], pact[lo:hi])
    assert torch.equal(y, part) and torch.equal(ya, part) and torch.equal(act, pact)


@pytest.mark.parametrize("B", [32768, 32769])
def test_deltas_match_fp64(B):
    """Deltas from the same activations in fp64, within the rounding of 64-term fp32 sums."""
    from paper_2010_12117_gb300 import binding
    p, x, t = _inputs(B)
    y = torch.empty(B, 2, device="cuda")
    act, delta = torch.empty(B, 128, device="cuda"), torch.empty(B, 130, device="cuda")
    g, loss = torch.empty(mlp.NPARAMS, device="cuda"), torch.empty(1, device="cuda")
    binding.mlp_forward(p, x, y, act)
    binding.mlp_backward(p, x, t, y, act, delta, g, loss)
    q = p.double()
    w2, w3 = q[576:576 + 4096].reshape(64, 64), q[4736:4736 + 128].reshape(2, 64)
    dy = (y.double() - t.double()) / B
    on = act.double() > 0
    dh2 = dy @ w3 * on[:, 64:]
    dh1 = dh2 @ w2 * on[:, :64]
    eps = 2.0 ** -24
    m0 = (y.abs() + t.abs()).double() / B  # sums of the terms' magnitudes
    m2 = m0 @ w3.abs()
    m1 = m2 @ w2.abs()
    # roundings: 2 of a difference and quotient, 3 more of two products and their sum, 64 more of 64 multiply-adds
    assert (delta[:, :2].double() - dy).abs().le(3 * eps * m0).all()
    assert (delta[:, 2:66].double() - dh2).abs().le(6 * eps * m2).all()
    assert (delta[:, 66:].double() - dh1).abs().le(72 * eps * m1).all()
