"""GPU tests of the float64 pair kernels' integer form (fixed64.cuh) and of its rule.

Scales: a box scaled by a power of two scales every coordinate exactly, and with it the integers and the results;
boxes beyond the rule's exponents take the float64 form for every pair.  All of them agree to 1e-12 (float64
rounding of sums over 27 N terms, amplified by their cancellation, is below 1e-13), charges, one-sided and
symmetric, and separate points, ball-trimmed or not, check points in one image list or in layers.

Near pairs: a pair within 2^-9 of the range takes float64, where differences of tiny coordinates are exact: pairs at
distances from either side of that line down to 1e-12, some at the origin with coordinates far below the
integers' unit, against the oracle's direct sums, to 1e-12 of each charge's own value (the pair's own terms, rounded
a few times, dominate it)."""
import numpy as np
import pytest

from oracle import psum_oracle as O
from paper_1310_4374_gb300 import binding as B
from paper_1310_4374_gb300 import workloads as W
from parity_check import assert_close

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def _run(x, q, d, y=None, **more):
    pc = B.PeriodicCoulomb(tuple(d), 8, 200, precision="fp64", **more)
    try:
        phi, g = pc(_dev(x), _dev(q)) if y is None else pc.at(_dev(x), _dev(q), _dev(y))
        return phi.cpu().numpy(), g.cpu().numpy()
    finally:
        pc.close()


FORMS = {"one-sided": dict(pairs="one-sided"), "symmetric": dict(pairs="symmetric"), "ball": dict(lam=1.6),
         "points": {}, "block_checks": dict(checks="points")}


@pytest.mark.parametrize("form", sorted(FORMS))
def test_power_of_two_scales(form):
    s = W.uniform_gauss(N=389, d=(1.0, 1.5, 2.0), p=8, M=200, seed=71)
    rng = np.random.default_rng(72)
    y = (rng.random((201, 3)) - 0.5) * np.array(s.d) if form == "points" else None
    ref = None
    for e in (0, -40, 25, 56, 59):          # 59: beyond the rule
        f = 2.0 ** e
        phi, g = _run(s.x * f, s.q, np.array(s.d) * f, None if y is None else y * f, **FORMS[form])
        if ref is None:
            ref = phi, g
        assert_close(phi * f, ref[0], 1e-12, f"{form} phi at 2^{e}")
        assert_close(g * f * f, ref[1], 1e-12, f"{form} grad at 2^{e}")


@pytest.mark.parametrize("form", ["one-sided", "symmetric"])
def test_power_of_two_charges(form):
    # charges beyond 2^+-200 take the float64 form, as do all of a charge's pairs beside ordinary ones
    s = W.uniform_gauss(N=389, d=(1.0, 1.5, 2.0), p=8, M=200, seed=74)
    q = s.q.copy()
    q[7::11] = 0.0
    q[3] = 0.0
    q[q != 0.0] -= q.sum() / np.count_nonzero(q)
    ref = _run(s.x, q, s.d, pairs=form)
    for e in (190, 240, -190, -240):
        f = 2.0 ** e
        phi, g = _run(s.x, q * f, s.d, pairs=form)
        assert_close(phi / f, ref[0], 1e-12, f"{form} phi, charges 2^{e}")
        assert_close(g / f, ref[1], 1e-12, f"{form} grad, charges 2^{e}")
    q[3] = 1e-150
    phi, g = _run(s.x, q, s.d, pairs=form)
    assert_close(phi, ref[0], 1e-12, f"{form} phi, one tiny charge")
    assert_close(g, ref[1], 1e-12, f"{form} grad, one tiny charge")


@pytest.mark.parametrize("pairs", ["one-sided", "symmetric"])
def test_near_pairs(pairs):
    rng = np.random.default_rng(73)
    n = 130
    d = (1.0, 1.0, 1.0)
    sep = np.concatenate([np.logspace(-12, -1, n - 30), 2.0 ** -7 * (1 + np.linspace(-0.3, 0.3, 30))])
    c = (rng.random((n, 3)) - 0.5) * 0.9
    c[::3] *= sep[::3, None]                  # a third of the pairs at the origin, at their own size
    u = rng.normal(size=(n, 3))
    u /= np.linalg.norm(u, axis=1)[:, None]
    x = np.concatenate([c + 0.5 * sep[:, None] * u, c - 0.5 * sep[:, None] * u])
    q = np.concatenate([np.ones(n), -np.ones(n)])
    phi, g = _run(x, q, d, pairs=pairs)
    ref = O.periodic_sum(x, q, d, 8, 200, parts=True)
    assert np.all(np.abs(phi - ref["phi"]) <= 1e-12 * np.maximum(np.abs(ref["phi"]), np.abs(ref["phi"]).min() + 1.0))
    gn = np.linalg.norm(ref["grad"], axis=1)
    assert np.all(np.linalg.norm(g - ref["grad"], axis=1) <= 1e-12 * gn)


@pytest.mark.parametrize("N", [47 * 128, 47 * 128 + 1, 48 * 128 + 127])
def test_symmetric_at_the_fourth_cta(N):
    # 47 and 48 tiles (three and four resident CTAs), full and ragged, against the one-sided kernel: the same
    # terms in another order (float64 rounding of 27 N terms)
    s = W.uniform_gauss(N=N, d=(1.0, 1.5, 2.0), p=8, M=200, seed=75)
    a, b = _run(s.x, s.q, s.d, pairs="symmetric"), _run(s.x, s.q, s.d, pairs="one-sided")
    assert_close(a[0], b[0], 1e-12, "phi")
    assert_close(a[1], b[1], 1e-12, "grad")
