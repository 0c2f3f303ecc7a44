"""The float64 packs' padding against charges and evaluation points that share its place, or the place (1000, 1000,
1000) of the float32 packs': both lie inside a box of side 4000, where every point counts as itself.  Sizes leave a
packed tile nearly empty or all but full.  The reference is the oracle in float64; sums over 27 N terms agree to the
float64 path's 1e-10 (Eq. st2), a point taken for another place is off by its own share of the sum, far above."""
import numpy as np
import pytest

from oracle import psum_oracle as O
from parity_check import assert_close
from paper_1310_4374_gb300 import binding as B
from paper_1310_4374_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-10
D = (4000.0, 4000.0, 4000.0)
FORMS = {"one-sided": dict(pairs="one-sided"), "symmetric": dict(pairs="symmetric"), "ball": dict(lam=1.6),
         "block_checks": dict(checks="points")}
PLACES = {"1000": (1000.0, 1000.0, 1000.0), "centre": (0.0, 0.0, 0.0)}


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def _system(N, place, seed=5):
    rng = np.random.default_rng(seed)
    x = rng.uniform(-0.5, 0.5, (N, 3)) * np.array(D)
    x[N // 3] = place
    q = rng.normal(size=N)
    q -= q.mean()
    return W.System(x, q, D, 8, 200, name=f"padding-{N}")


@pytest.mark.parametrize("place", sorted(PLACES))
@pytest.mark.parametrize("N", [129, 255])
@pytest.mark.parametrize("form", sorted(FORMS))
def test_charge_at_the_paddings_place(form, N, place):
    s = _system(N, PLACES[place])
    pc = B.PeriodicCoulomb(D, s.p, s.M, precision="fp64", **FORMS[form])
    try:
        x, q = _dev(s.x), _dev(s.q)
        phi, g = (t.cpu().numpy() for t in pc(x, q))
        gphi, gg = torch.empty_like(q), torch.empty_like(x)
        B.psum_eval_graph(pc.plan, x, q, gphi, gg, check=True)
    finally:
        pc.close()
    ref = O.periodic_sum(s.x, s.q, D, s.p, s.M, lam=FORMS[form].get("lam", 0.0))
    assert_close(phi, ref["phi"], TOL, "phi")
    assert_close(g, ref["grad"], TOL, "grad")
    assert np.array_equal(gphi.cpu().numpy(), phi) and np.array_equal(gg.cpu().numpy(), g)


@pytest.mark.parametrize("place", sorted(PLACES))
@pytest.mark.parametrize("charge_there", [False, True])
def test_point_at_the_paddings_place(charge_there, place):
    s = _system(129, PLACES[place] if charge_there else (123.0, -456.0, 789.0))
    y = np.random.default_rng(6).uniform(-0.5, 0.5, (130, 3)) * np.array(D)
    y[77] = PLACES[place]
    pc = B.PeriodicCoulomb(D, s.p, s.M, precision="fp64")
    try:
        phi, g = (t.cpu().numpy() for t in pc.at(_dev(s.x), _dev(s.q), _dev(y)))
    finally:
        pc.close()
    ref = O.Plan(D, s.p, s.M).evaluate(s.x, s.q, targets=y, parts=True)
    assert_close(phi, ref["phi"], TOL, "phi")
    assert_close(g, ref["grad"], TOL, "grad")


@pytest.mark.parametrize("place", sorted(PLACES))
def test_backward_with_a_charge_at_the_paddings_place(place):
    from paper_1310_4374_gb300.autograd import PeriodicCoulombEnergy

    s = _system(129, PLACES[place])
    ref = O.energy_and_gradients(O.Plan(D, s.p, s.M), s.x, s.q)
    mod = PeriodicCoulombEnergy(D, s.p, s.M, precision="fp64")
    try:
        x, q = _dev(s.x).requires_grad_(), _dev(s.q).requires_grad_()
        E = mod(x, q)
        E.backward()
        assert abs(E.item() - ref["E"]) <= 10 * TOL * abs(ref["E"])
        assert_close(x.grad.cpu().numpy(), ref["dEdx"], TOL, "dEdx")
        gq = q.grad.cpu().numpy()               # up to a constant on the neutral subspace
        assert_close(gq - gq.mean(), ref["dEdq"] - ref["dEdq"].mean(), TOL, "dEdq")
    finally:
        mod.close()


@pytest.mark.parametrize("place", sorted(PLACES))
def test_batch_with_a_charge_at_the_paddings_place(place):
    systems = [_system(129, PLACES[place], seed=7), _system(255, PLACES[place], seed=8)]
    pb = B.PeriodicBatch(systems, precision="fp64")
    try:
        phi, g = (t.cpu().numpy() for t in pb(_dev(np.concatenate([s.x for s in systems])),
                                              _dev(np.concatenate([s.q for s in systems]))))
        for b, s in enumerate(systems):
            sl = slice(pb.offsets[b], pb.offsets[b + 1])
            ref = O.periodic_sum(s.x, s.q, D, s.p, s.M)
            assert_close(phi[sl], ref["phi"], TOL, f"phi of {b}")
            assert_close(g[sl], ref["grad"], TOL, f"grad of {b}")
    finally:
        pb.close()
