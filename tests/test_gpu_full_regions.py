"""GPU parity of colour phases whose regions hold more beads than shared memory stages: by groups of
blocks through the global cell lists where that is the layer's average (blocks of a group evaluate a
queue's moves ahead of their turn), by one warp where it is a rare dense region. Chains fill one
octant of the box, so queues of one phase range from empty to thousands of beads; bonds and supports
cross the region borders (deferrals)."""
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


def octant(n_chains, length, phi, seed):
    """Chains of a periodic cube unwrapped into a box of twice its side."""
    s = I.make_system([length] * n_chains, 0, I.box_for_volume_fraction(n_chains * length, phi), seed=seed)
    x = s.pos.reshape(n_chains, length, 3)
    d = np.diff(x, axis=1)
    d -= s.box_L * np.round(d / s.box_L)
    x = np.concatenate([x[:, :1], x[:, :1] + np.cumsum(d, axis=1)], axis=1).reshape(-1, 3)
    L = 2.0 * s.box_L
    return I.System(np.minimum(np.mod(x, L), np.nextafter(L, 0.0)), s.chain_len, L)


@pytest.mark.parametrize("n_chains, grid, K, precision", [
    (225, 2, 2, wmcd.FP64), (225, 2, 2, wmcd.MIXED), (225, 3, 3, wmcd.FP64), (225, 3, 3, wmcd.MIXED),
    (700, 4, 2, wmcd.MIXED),                                             # eight groups of blocks
    (225, 4, 2, wmcd.FP64), (225, 4, 2, wmcd.MIXED)])                    # one dense region of eight
def test_regions_beyond_staging(n_chains, grid, K, precision):
    s = octant(n_chains, 20, 0.1 if n_chains > 300 else 0.2, seed=41)
    p = wmcd.default_params(s.n_beads, s.box_L, seed=19, precision=precision, colour_K=K, n_cap=12)
    p["grid_layer"] = [grid] + [0] * 15
    gpu, ref = run_pair(p, s, 1)
    a = gpu.trace(0)[0]
    ran = ((a & 3) != 0) & ((a & 4) == 0)
    assert ran.sum() > 0.3 * len(a) and (grid == K or ((a & 4) != 0).any())
