"""GPU parity of the shared-memory serial phase at the edges of its ranges: block sizes (320, 1,024
and 2,048 beads), groups of 32 beads, supports and candidate lists on both sides of what one warp
holds, beads in no spatial order, and bonds across groups. Every decision against the oracle."""
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


def params(s, precision, **kw):
    p = wmcd.default_params(s.n_beads, s.box_L, seed=17, precision=precision, serial_only=True, **kw)
    assert not any(p["grid_layer"])
    return p


@pytest.mark.parametrize("precision", [wmcd.FP64, wmcd.MIXED])
@pytest.mark.parametrize("n", [2, 31, 32, 33, 319, 320, 321, 1023, 1024, 1025, 2047, 2048])
def test_chain_lengths(n, precision):
    L = max(40.0, I.box_for_volume_fraction(n, 1e-3))
    s = I.single_chain(n, L, seed=n)
    run_pair(params(s, precision, planewave_mode=wmcd.PLANEWAVE_PERIODIC), s, 3 if n < 1000 else 1)


@pytest.mark.parametrize("precision", [wmcd.FP64, wmcd.MIXED])
@pytest.mark.parametrize("n", [300, 1500])
def test_dense_chains_overflow_a_warp(n, precision):
    """Volume fraction 0.2: the second layer's supports (about 25-200 beads) and their candidates
    pass the 48 and 160 that one warp holds, so moves change between a warp and the block."""
    s = I.make_system([n // 10] * 10, 0, I.box_for_volume_fraction(n, 0.2), seed=5)
    gpu, ref = run_pair(params(s, precision, A0=0.3), s, 2)
    na = gpu.trace(1)[1]
    assert (na > 48).any() and (na < 48).any()


@pytest.mark.parametrize("precision", [wmcd.FP64, wmcd.MIXED])
def test_spheres_in_a_well_glauber(precision):
    """Free spheres: no bead order to speak of, every group's ball spans the box."""
    s = I.free_spheres(700, 5e-3, seed=9)
    run_pair(params(s, precision, ext_kappa=0.002, acceptance=wmcd.ACCEPT_GLAUBER, bond_type=wmcd.BOND_NONE), s, 3)


def test_uniform_centres_dilute():
    """Centres uniform in a dilute box: A_w from a mean support below one bead, so displacements are
    several times those of a bead-centred move of the same scale."""
    s = I.single_chain(200, 100.0, seed=3)
    run_pair(params(s, wmcd.MIXED, centring=wmcd.CENTRE_UNIFORM, A0=0.2), s, 10)
