"""A batch whose colour phases hold more queues than the GPU runs at once, though each member's alone are
few: its launch shapes are not those of a lone member, its trajectories are."""
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
def test_members_follow_their_lone_trajectories(precision):
    systems = [I.dilute_chains(40 + k % 3, 64, 1e-3, seed=k) for k in range(48)]
    params = [wmcd.default_params(s.n_beads, s.box_L, seed=5, sim_id=k, precision=precision) for k, s in enumerate(systems)]
    assert sum((p["grid_layer"][0] // 2) ** 3 for p in params) > 16 * 152
    b = wmcd.Batch(len(params), sum(wmcd.batch_need(p) for p in params) + (1 << 20))
    slots = [b.admit(p, s.pos, s.chain_len) for p, s in zip(params, systems)]
    b.step(3)
    for k in (0, 1, 2, 23, 47):
        sim = wmcd.Simulation(params[k], systems[k].pos, systems[k].chain_len)
        sim.sweep(3)
        m = b.sim(slots[k])
        assert np.array_equal(m.positions(unwrapped=True), sim.positions(unwrapped=True))
        x, y = m.stats(), sim.stats()
        assert x.error_flags == 0 and list(x.accepts) == list(y.accepts) and list(x.deferred) == list(y.deferred)
        sim.close()
    b.close()
