"""The binary32 screen of whole-GPU moves in a box far larger than the cutoff (L = 10^4 r_c, coordinates
of eight digits in the first unit): pairs just inside the cutoff that their binary32 distances put outside count
in the binary64 energy change as in the one-block form and the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_1611_09160_gb300 import wmcd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    wmcd.build()
    wmcd.load()


@pytest.mark.parametrize("unit", [10.0, 1e-3])
def test_pairs_at_the_cutoff_of_a_huge_box(unit):
    rng = np.random.default_rng(3)
    L, rc, pairs = 1e7 * unit, 1e3 * unit, 1200
    site = rng.choice(40 ** 3, pairs, replace=False)
    a = 8.5e6 + 2e4 * np.stack([site % 40, site // 40 % 40, site // 1600], axis=1) + rng.uniform(0.0, 5e3, (pairs, 3))
    u = rng.normal(size=(pairs, 3))
    u /= np.linalg.norm(u, axis=1)[:, None]
    pos = np.stack([a, a + rng.uniform(998.0, 1000.0, (pairs, 1)) * u], axis=1).reshape(-1, 3) * unit
    n = 2 * pairs
    p = wmcd.default_params(n, L, lambda_min=4e5 * unit, lambda_max=1.2e6 * unit, A0=0.01, wca_sigma=rc / 2.0 ** (1.0 / 6.0),
                            bond_type=wmcd.BOND_NONE, seed=4, serial_only=True)
    p["grid_f"] = 128
    one = np.ones(n, np.int32)
    big = wmcd.Simulation(dict(p, big_support=1), pos, one)
    ref = wmcd.Simulation(dict(p, big_support=-1), pos, one)
    o = O.Oracle(dict(p, big_support=-1), pos, one)
    big.profile(True)
    big.sweep(1)
    ref.sweep(1)
    o.sweep_sample(60)
    assert big.kernel_times()["whole_gpu_serial"][0] > 0
    want, got = ref.trace_du(0), big.trace_du(0)
    assert np.abs(want).max() > 1e-6
    assert np.abs(o.trace_du(0)[:60] - want[:60]).max() <= 1e-9
    assert np.abs(got - want).max() <= 1e-9
    assert big.stats().partner_evals == ref.stats().partner_evals
