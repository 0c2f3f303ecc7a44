"""The spatial order by counting and by radix passes, at the sizes where either can go wrong: a few
points, blocks of four keys and of 32 points with remainders, one key shared by every point, and
both sides of the size where the radix sort takes over.  A wrong or incomplete permutation drops
charges, so float32 results (in that order) against float64 ones (in the caller's order) show it.
The tolerance is the float32 path's 1e-6 (Eq. st2); charges in one cell of the key grid are 2^-8 of
the box apart, far above what float32 offsets resolve."""
import numpy as np
import pytest

from parity_check import assert_close
from paper_1310_4374_gb300 import binding as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

D = (1.0, 1.5, 2.0)


def _run(precision, x, q):
    pc = B.PeriodicCoulomb(D, 8, 200, precision=precision, mean="none")
    try:
        phi, grad = pc(torch.as_tensor(x, device="cuda:0"), torch.as_tensor(q, device="cuda:0"))
        return phi.cpu().numpy(), grad.cpu().numpy()
    finally:
        pc.close()


@pytest.mark.parametrize("N", [2, 3, 31, 33, 127, 513, 4099, 4865, 9729, 14593, 24320, 24321])
@pytest.mark.parametrize("one_cell", [False, True])
def test_order_keeps_every_charge(N, one_cell):
    rng = np.random.default_rng(N)
    x = rng.uniform(-0.5, 0.5, (N, 3)) * np.asarray(D)
    if one_cell and N <= 4099:
        x = 0.01 * np.asarray(D) + x / 256.0 * 0.9 / 2      # inside one cell of the 256^3 grid or its neighbours
    q = rng.normal(size=N)
    q -= q.mean()
    phi, grad = _run("fp32c", x, q)
    ref_phi, ref_grad = _run("fp64", x, q)
    # the terms' own size scales the error: 1/r sums of a small cluster cancel less than its net charge
    assert_close(phi, ref_phi, 1e-6, "phi")
    assert_close(grad, ref_grad, 1e-6, "grad")
