"""The energy change of a plane wave is summed in an order that the state alone fixes: a move decided
within rounding of its threshold comes out the same on every run. The threshold kT (-ln(1 - u)) is moved
onto the energy change by bisection over kT (neither the draw nor the energies depend on it), then the
move is repeated at every kT within a few units of the last place."""
import math

import numpy as np
import pytest

from paper_1611_09160_gb300 import inputs as I
from paper_1611_09160_gb300 import wmcd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    wmcd.build()
    wmcd.load()


@pytest.mark.parametrize("precision", [wmcd.FP64, wmcd.MIXED])
@pytest.mark.parametrize("phi, A0", [(0.1, 0.5), (0.02, 40.0)])      # the second: long reach, full columns
def test_decision_at_a_tie_repeats(phi, A0, precision):
    s = I.dilute_chains(200, 41, phi, seed=3)
    p = wmcd.default_params(s.n_beads, s.box_L, seed=6, precision=precision, A0=A0,
                            planewave_mode=wmcd.PLANEWAVE_PERIODIC)

    def accepted(kT):
        sim = wmcd.Simulation(dict(p, kT=kT), s.pos, s.chain_len)
        sim.planewave(1)
        out, mode = sim.trace(-1)
        assert sim.stats().error_flags == 0
        sim.close()
        return int(out[0]) == 1

    lo, hi = 1e-6, 1e12
    assert not accepted(lo) and accepted(hi)
    while math.nextafter(lo, math.inf) < hi:
        mid = math.sqrt(lo * hi) if hi > 2.0 * lo else 0.5 * (lo + hi)
        mid = min(max(mid, math.nextafter(lo, math.inf)), math.nextafter(hi, 0.0))
        if accepted(mid):
            hi = mid
        else:
            lo = mid
    kT = hi
    for _ in range(24):
        kT = math.nextafter(kT, 0.0)
    for step in range(48):
        got = {accepted(kT) for _ in range(8)}
        assert len(got) == 1, f"kT = {kT!r}: the same move was both accepted and rejected"
        kT = math.nextafter(kT, math.inf)
