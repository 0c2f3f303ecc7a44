"""The spatial order where every point has the same key: all inside one cell of the 256^3 grid, so that the index alone
decides each place.  One size for each number of points a lane that the order by counting takes (1 to 5, with
remainders) and either side of the size where the radix sort takes over.  A wrong or incomplete permutation drops
or doubles charges, so float32 results (in that order) against float64 ones (in the caller's) show it, to the
float32 path's 1e-6 (Eq. st2)."""
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


@pytest.mark.parametrize("N", [130, 4865, 9729, 14593, 19457, 24320, 24321])
def test_one_key_for_every_point(N):
    rng = np.random.default_rng(N)
    cell = (131 + rng.uniform(0.05, 0.95, (N, 3))) / 256.0 - 0.5
    assert np.all(np.floor((cell + 0.5) * 256.0) == 131)
    x = cell * np.asarray(D)
    q = rng.normal(size=N)
    q -= q.mean()
    phi, grad = _run("fp32c", x, q)
    ref_phi, ref_grad = _run("fp64", x, q)
    assert_close(phi, ref_phi, 1e-6, "phi")
    assert_close(grad, ref_grad, 1e-6, "grad")
