"""Device memory of a lone simulation: one whose layers all run in shared memory (or on the whole GPU)
holds no scratch for the blocks of the speculative serial phase, so it takes what it takes in a batch."""
import pytest

from paper_1611_09160_gb300 import inputs as I
from paper_1611_09160_gb300 import wmcd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    wmcd.build()
    wmcd.load()


@pytest.mark.parametrize("n, extra", [(33, {}), (2048, {}), (1000, {"big_support": 50})])
def test_all_serial_simulation(n, extra):
    s = I.single_chain(n, I.box_for_volume_fraction(n, 1e-2), seed=1)
    p = dict(wmcd.default_params(s.n_beads, s.box_L, precision=wmcd.MIXED, serial_only=True), **extra)
    sim = wmcd.Simulation(p, s.pos, s.chain_len)
    assert sim.device_bytes() <= wmcd.batch_need(p)          # a batch rounds every array up
    sim.sweep(2)
    assert sim.stats().error_flags == 0
