"""The far field and the moments by columns of the expansion, with the gradient's own coefficients,
at the degrees where the sharing of columns or the memory can go wrong: the lowest, odd and even ones,
the last degree whose moments are summed by columns and the first that is not, and one whose tables
pass the default shared memory; point counts that end inside a block.  Against the oracle at the
float64 paths' 1e-10 (Eq. st2)."""
import numpy as np
import pytest

from oracle import psum_oracle as O
from parity_check import assert_close
from paper_1310_4374_gb300 import binding as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

D = (1.0, 1.25, 1.5)


def _system(N, seed=0):
    rng = np.random.default_rng(seed)
    x = rng.uniform(-0.5, 0.5, (N, 3)) * np.asarray(D)
    q = rng.normal(size=N)
    return x, q - q.mean()


@pytest.mark.parametrize("p, M, N", [(1, 12, 2), (2, 20, 33), (3, 40, 64), (7, 150, 31), (8, 200, 257), (13, 450, 100),
                                     (31, 1400, 65)])
@pytest.mark.parametrize("precision", ["fp64", "ff"])
def test_far_field(p, M, N, precision):
    x, q = _system(N, p)
    ref = O.periodic_sum(x, q, D, p, M)
    pc = B.PeriodicCoulomb(D, p, M, precision=precision)
    try:
        xt, qt = torch.as_tensor(x, device="cuda:0"), torch.as_tensor(q, device="cuda:0")
        phi, grad = pc(xt, qt)
        phi_only, _ = pc(xt, qt, grad=False)
    finally:
        pc.close()
    assert_close(phi.cpu().numpy(), ref["phi"], 1e-10, "phi")
    assert_close(grad.cpu().numpy(), ref["grad"], 1e-10, "grad")
    assert torch.equal(phi_only, phi)


@pytest.mark.parametrize("p, M, N", [(1, 12, 2), (2, 20, 33), (9, 250, 700), (25, 950, 65), (26, 1000, 65), (27, 1100, 65)])
def test_moments(p, M, N):
    x, q = _system(N, 100 + p)
    ref = O.energy_and_gradients(O.Plan(D, p, M), x, q)
    plan = B.psum_plan_create_ex(D, p, M, "fp64")
    try:
        xt, qt = torch.as_tensor(x, device="cuda:0"), torch.as_tensor(q, device="cuda:0")
        phi, dEdq = torch.empty_like(qt), torch.empty_like(qt)
        grad, dEdx = torch.empty_like(xt), torch.empty_like(xt)
        B.psum_eval(plan, xt, qt, phi, grad, check=True)
        B.psum_energy_backward(plan, xt, qt, phi, grad, None, dEdq, dEdx)
        torch.cuda.synchronize()
    finally:
        B.psum_destroy(plan)
    assert_close(dEdq.cpu().numpy(), ref["dEdq"], 1e-10, "dEdq")
    assert_close(dEdx.cpu().numpy(), ref["dEdx"], 1e-10, "dEdx")
