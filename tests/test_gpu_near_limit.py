"""The float64 pair sums at the lower end of their range: the estimate of 1/r takes squared distances from 2^-126
on.  Charges within 2^-63.5 of each other count as coincident (K(0) = 0), from there to 2^-63 an evaluation is refused as not
finite, from 2^-63 on the pair counts; in a box of that size too, and not where the other one is no charge but a
pack's padding at the centre of the box.  Values against exact coincidence or the oracle, to the float64 path's 1e-10."""
import numpy as np
import pytest

from oracle import psum_oracle as O
from parity_check import assert_close
from paper_1310_4374_gb300 import binding as B
from paper_1310_4374_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

D = (1.0, 1.5, 2.0)
TOL = 1e-10
NOT_FINITE = B.PSUM_ERR_NONFINITE


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def _run(x, q, d=D, y=None, **more):
    pc = B.PeriodicCoulomb(tuple(d), 8, 200, precision="fp64", **more)
    try:
        phi, g = pc(_dev(x), _dev(q)) if y is None else pc.at(_dev(x), _dev(q), _dev(y))
        return phi.cpu().numpy(), g.cpu().numpy()
    finally:
        pc.close()


def _system(first, second):
    s = W.uniform_gauss(N=130, d=D, p=8, M=200, seed=76)
    s.x[40] = (first, 0.0, 0.0)
    s.x[90] = (second, 0.0, 0.0)
    return s


@pytest.mark.parametrize("pairs", ["one-sided", "symmetric"])
def test_pairs_at_the_end_of_the_range(pairs):
    # 0.25 and -0.25 of an octave about 2^-63.5 and 2^-63, across the origin
    def at(e):
        s = _system(0.5 * 2.0 ** e, -0.5 * 2.0 ** e)
        return _run(s.x, s.q, pairs=pairs)

    s = _system(0.0, 0.0)
    ref = _run(s.x, s.q, pairs=pairs)
    phi, g = at(-63.75)
    assert_close(phi, ref[0], TOL, "phi")
    assert_close(g, ref[1], TOL, "grad")
    with pytest.raises(B.PsumError) as e:
        at(-63.25)
    assert e.value.status == NOT_FINITE
    phi, g = at(-62.75)
    r = 2.0 ** -62.75
    assert abs(phi[40] * r - s.q[90]) <= TOL and abs(phi[90] * r - s.q[40]) <= TOL
    assert abs(g[40, 0] * r * r + s.q[90]) <= TOL and abs(g[90, 0] * r * r - s.q[40]) <= TOL


def test_point_at_the_end_of_the_range():
    s = _system(0.0, 0.3)
    y = np.array([[2.0 ** -63.25, 0.0, 0.0], [0.1, 0.2, 0.3]])
    with pytest.raises(B.PsumError) as e:
        _run(s.x, s.q, y=y)
    assert e.value.status == NOT_FINITE


@pytest.mark.parametrize("pairs", ["one-sided", "symmetric"])
def test_padding_is_no_charge(pairs):
    # 130 charges leave padding at the centre of the box; charges in the refused distance of it
    s = _system(2.0 ** -63.25, 0.25)
    phi, g = _run(s.x, s.q, pairs=pairs)
    ref = O.periodic_sum(s.x, s.q, D, s.p, s.M)
    assert_close(phi, ref["phi"], TOL, "phi")
    assert_close(g, ref["grad"], TOL, "grad")


@pytest.mark.parametrize("pairs", ["one-sided", "symmetric"])
def test_box_of_the_range(pairs):
    # hundreds of pairs in the refused half octave, in a box the integers could hold
    s = W.uniform_gauss(N=389, d=D, p=8, M=200, seed=71)
    with pytest.raises(B.PsumError) as e:
        _run(s.x * 2.0 ** -60, s.q, np.array(D) * 2.0 ** -60, pairs=pairs)
    assert e.value.status == NOT_FINITE
