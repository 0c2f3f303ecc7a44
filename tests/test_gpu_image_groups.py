"""The image groups of the symmetric FP32C kernel at the sizes where the rule turns: three images a group with the
fast terms from 13 tiles on, one with the refined terms up to four items a CTA.  Each size against the oracle on
sampled charges at the path's 1e-6 (Eq. st2), full and ragged last tiles."""
import numpy as np
import pytest

from oracle import psum_oracle as O
from paper_1310_4374_gb300 import binding as B
from paper_1310_4374_gb300 import workloads as W
from parity_check import assert_close

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("terms, N, groups", [("fast", 6145, 9), ("fast", 12288, 9), ("refined", 8000, 27), ("refined", 12289, 9)])
def test_groups(terms, N, groups):
    s = W.uniform_gauss(N=N, d=(1.0, 1.5, 2.0), p=8, M=200, seed=81)
    pc = B.PeriodicCoulomb(s.d, s.p, s.M, precision="fp32c", terms=terms)
    try:
        assert B.psum_pair_kernel(pc.plan, N) == ("symmetric", groups)
        phi, g = (t.cpu().numpy() for t in pc(torch.as_tensor(s.x, device="cuda"), torch.as_tensor(s.q, device="cuda")))
    finally:
        pc.close()
    k = np.sort(np.random.default_rng(1).choice(N, size=512, replace=False))
    ref = O.Plan(s.d, s.p, s.M).evaluate(s.x, s.q, targets=s.x[k])
    assert_close(phi[k], ref["phi"], 1e-6, "phi")
    assert_close(g[k], ref["grad"], 1e-6, "grad")
