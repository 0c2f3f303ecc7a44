"""The float32 packs' padding in far units: a last group of 16 charges about its midpoint, the rest padding, and
a dense cluster in another group with a charge at (1000, 1000, 1000) from that midpoint, exact in float32, in a box of side
4000.  Padding is no charge wherever it lies, as a source and as a target of the reactions.  Tolerances: the
precisions' own against the float64 sums (1e-6 and 1e-10, Eq. st2)."""
import numpy as np
import pytest

from parity_check import assert_close
from paper_1310_4374_gb300 import binding as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

D = (4000.0, 4000.0, 4000.0)
TOL = {"fp32c": 1e-6, "ff": 1e-10}


def _run(x, q, **kw):
    pc = B.PeriodicCoulomb(D, 8, 200, **kw)
    try:
        phi, g = pc(torch.as_tensor(x, device="cuda"), torch.as_tensor(q, device="cuda"))
        return phi.cpu().numpy(), g.cpu().numpy()
    finally:
        pc.close()


def _grid(n):
    a = np.arange(-7, 8)
    g = np.stack(np.meshgrid(a, a, a, indexing="ij"), -1).reshape(-1, 3).astype(float)
    return g[np.argsort((g ** 2).sum(1), kind="stable")][:n]


@pytest.mark.parametrize("pairs", ["one-sided", "symmetric"])
@pytest.mark.parametrize("lam", [0.0, 1.6])
@pytest.mark.parametrize("precision", ["fp32c", "ff"])
@pytest.mark.parametrize("dense", [512, 1024, 1536])
def test_padding_in_a_far_unit(dense, precision, lam, pairs):
    if lam and pairs == "symmetric":
        pytest.skip("ball-trimmed plans are one-sided")
    base = np.array((500.0, -1500.0, 250.0))         # late on the curve: the small cluster is the last group
    half = _grid(23)[1:12] * 4.0
    small = np.unique(np.concatenate([half, -half]), axis=0) + base
    x = np.concatenate([_grid(dense) * 6.0 + base + 1000.0, small])
    q = np.random.default_rng(dense).normal(size=len(x))
    q -= q.mean()
    phi, g = _run(x, q, precision=precision, pairs=pairs, lam=lam)
    ref = _run(x, q, precision="fp64", lam=lam)
    assert_close(phi, ref[0], TOL[precision], "phi")
    assert_close(g, ref[1], TOL[precision], "grad")
