"""GPU parity of the serial phase whose moves are evaluated ahead of their turn by the blocks of a
cooperative launch (a lone simulation): every decision and position must be that of the moves run
one after another. The cases reach each rule of the window walk: moves that conflict with an
accepted one, runs of rejections and of acceptances, windows longer than the slots left, lists of
deferred slots, supports beyond a block's scratch, and bonds much longer than a support."""
import numpy as np
import pytest

from paper_1611_09160_gb300 import inputs as I
from paper_1611_09160_gb300 import wmcd

from test_gpu_parity import run_pair

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    wmcd.build()
    wmcd.load()


@pytest.mark.parametrize("precision", [wmcd.FP64, wmcd.MIXED])
@pytest.mark.parametrize("A0", [0.02, 0.5, 2.0])
def test_runs_of_acceptances_and_rejections(precision, A0):
    """2,304 chain beads (above the shared-memory serial phase), every layer serial: acceptance from
    nearly all to nearly none, conflicts in a box of a few supports."""
    s = I.make_system([48] * 48, 0, I.box_for_volume_fraction(2304, 0.02), seed=31)
    p = wmcd.default_params(s.n_beads, s.box_L, seed=3, precision=precision, A0=A0, serial_only=True)
    p["big_support"] = -1
    gpu, ref = run_pair(p, s, 2)
    st = ref.stats()
    f = st.accepted_total / max(1, sum(st.attempts))
    assert f > 0.9 if A0 < 0.1 else f < 0.9


@pytest.mark.parametrize("precision", [wmcd.FP64, wmcd.MIXED])
def test_supports_beyond_a_block(precision):
    """4,608 chain beads under scales of 0.46-0.5 box sides: supports on both sides of the 2,048
    members a block's scratch holds, against the one-block form (128 threads), which the other
    parity tests compare with the oracle (too slow for such supports)."""
    s = I.make_system([32] * 144, 0, I.box_for_volume_fraction(4608, 0.15), seed=15)
    p = wmcd.default_params(s.n_beads, s.box_L, seed=6, precision=precision, serial_only=True,
                            lambda_min=0.46 * s.box_L, planewave_mode=wmcd.PLANEWAVE_PERIODIC)
    p["big_support"] = -1
    a, b = (wmcd.Simulation(p, s.pos, s.chain_len) for _ in range(2))
    b.set_block(2, 128)
    a.sweep(1)
    b.sweep(1)
    n = a.trace(0)[1]
    assert (n > 2048).any() and (n < 2048).any() and 0 < a.stats().accepts[0] < a.stats().attempts[0]
    assert np.array_equal(a.trace(0)[0], b.trace(0)[0]) and np.array_equal(n, b.trace(0)[1])
    assert np.array_equal(a.positions(unwrapped=True), b.positions(unwrapped=True))


@pytest.mark.parametrize("n", [1, 2, 3, 17])
def test_fewer_slots_than_the_window(n):
    """A handful of free beads in a wide well (no chain to overlap): most layers have no slot or one."""
    L = 64.0
    pos = np.random.default_rng(5).random((n, 3)) * L * 0.999
    s = I.System(pos, np.ones(n, np.int32), L)
    p = wmcd.default_params(n, L, seed=8, bond_type=wmcd.BOND_NONE, wca_eps=0.0, ext_kappa=0.01)
    run_pair(p, s, 40, trace_every=7)


def test_bonds_longer_than_the_supports():
    """Soft bonds of rest length 30 between beads of neighbouring rows: a move reads partners far
    outside its own ball, which an earlier move of the window may have shifted."""
    rng = np.random.default_rng(7)
    n, L = 2400, 160.0
    pos = rng.random((n, 3)) * L
    pos = np.minimum(pos, np.nextafter(L, 0.0))
    s = I.System(pos, np.full(n // 8, 8, np.int32), L)
    p = wmcd.default_params(n, L, seed=12, bond_k=0.02, bond_r0=30.0, wca_eps=0.0, precision=wmcd.MIXED,
                            serial_only=True, lambda_max=24.0)
    gpu, ref = run_pair(p, s, 2)
    assert 0 < gpu.stats().accepted_total
