"""The energy change of a plane wave is summed in an order that the state alone fixes: a move decided
within rounding of its threshold comes out the same on every run. The threshold kT (-ln(1 - u)) is moved
onto the energy change by bisection over kT (neither the draw nor the energies depend on it), then the
move is repeated at every kT within a few units of the last place. The kT found is also the oracle's."""
import math

import pytest

import oracle as O
from paper_1611_09160_gb300 import inputs as I
from paper_1611_09160_gb300 import wmcd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    wmcd.build()
    wmcd.load()


def first_move(p, s, kT):
    sim = wmcd.Simulation(dict(p, kT=kT), s.pos, s.chain_len)
    sim.planewave(1)
    out, mode = sim.trace(-1)
    assert sim.stats().error_flags == 0
    sim.close()
    return int(out[0]) == 1


def tie(p, s):
    """The smallest kT at which the first plane wave is accepted."""
    lo, hi = 1e-6, 1e12
    assert not first_move(p, s, lo) and first_move(p, s, hi)
    while math.nextafter(lo, math.inf) < hi:
        mid = math.sqrt(lo * hi) if hi > 2.0 * lo else 0.5 * (lo + hi)
        mid = min(max(mid, math.nextafter(lo, math.inf)), math.nextafter(hi, 0.0))
        if first_move(p, s, mid):
            hi = mid
        else:
            lo = mid
    return hi


# the second: a reach of several cells, most beads with more partners than a column holds
@pytest.mark.parametrize("precision", [wmcd.FP64, wmcd.MIXED])
@pytest.mark.parametrize("phi, A0", [(0.1, 0.5), (0.02, 40.0)])
def test_decision_at_a_tie(phi, A0, precision):
    s = I.dilute_chains(200, 41, phi, seed=3)
    p = wmcd.default_params(s.n_beads, s.box_L, seed=6, precision=precision, A0=A0,
                            planewave_mode=wmcd.PLANEWAVE_PERIODIC)
    at = tie(p, s)
    for rel, accepts in ((-1e-9, 2), (1e-9, 1)):       # binary64 energies: equal to rounding
        o = O.Oracle(dict(p, kT=at * (1.0 + rel)), s.pos, s.chain_len)
        o.planewave(1)
        assert int(o.trace_pw()[0][0]) == accepts
        o.close()
    kT = at
    for _ in range(24):
        kT = math.nextafter(kT, 0.0)
    for step in range(48):
        got = {first_move(p, s, kT) for _ in range(8)}
        assert len(got) == 1, f"kT = {kT!r}: the same move was both accepted and rejected"
        kT = math.nextafter(kT, math.inf)
