"""Colour phases of more queues than one block scans (over 32,768 buckets and regions: scans by several
blocks, the lists of dense regions filled by all of them, region counters in global memory), decision by
decision against the oracle: a large box with few beads, most of them in blobs of every tier's density in
different parts of the box, so that each block's share has entries for both lists."""
import numpy as np
import pytest

from paper_1611_09160_gb300 import inputs as I
from paper_1611_09160_gb300 import wmcd

from test_gpu_parity import run_pair

pytestmark = pytest.mark.gpu

L = 1600.0
SIDE = L / 33                                          # regions of one colour, a quarter side off the origin


@pytest.fixture(scope="module", autouse=True)
def built():
    wmcd.build()
    wmcd.load()


def blobs():
    """Chains of five; (chains, volume fraction, region) of each blob, the rest anywhere."""
    spec = [(180, 0.2, (3, 17, 1)), (60, 0.05, (12, 3, 9)), (180, 0.2, (25, 1, 17)), (40, 0.03, (20, 22, 24)),
            (175, 0.2, (32, 32, 31)), (25, 0.02, (7, 0, 14))]
    parts, lens = [], []
    for k, (n, phi, region) in enumerate(spec):
        b = I.make_system([5] * n, 0, I.box_for_volume_fraction(5 * n, phi), seed=50 + k)
        x = b.pos.reshape(n, 5, 3)
        d = np.diff(x, axis=1)
        d -= b.box_L * np.round(d / b.box_L)
        x = np.concatenate([x[:, :1], x[:, :1] + np.cumsum(d, axis=1)], axis=1).reshape(-1, 3)
        parts.append(np.mod(x + SIDE / 4 + SIDE * np.array(region) + 0.5 * (SIDE - b.box_L), L))
        lens.append(b.chain_len)
    rest = I.make_system([5] * 40, 0, L, seed=9)
    pos = np.concatenate(parts + [rest.pos])
    return I.System(np.minimum(pos, np.nextafter(L, 0.0)), np.concatenate(lens + [rest.chain_len]), L)


@pytest.mark.parametrize("precision, level2", [(wmcd.FP64, 0), (wmcd.MIXED, 0), (wmcd.MIXED, 1)])
def test_scans_by_several_blocks(precision, level2):
    s = blobs()
    p = wmcd.default_params(s.n_beads, L, seed=23, precision=precision, lambda_max=12.0, n_cap=8, level2=level2)
    p["grid_f"] = 264
    p["grid_layer"] = [66, 34] + [0] * 14
    counts = np.zeros(33 ** 3, int)                    # beads per region of the last colour, near enough
    c = (np.mod(s.pos - SIDE / 4, L) / SIDE).astype(int) % 33
    np.add.at(counts, c[:, 0] + 33 * (c[:, 1] + 33 * c[:, 2]), 1)
    share = np.arange(33 ** 3) // 8192
    for lo, hi in ((81, 640), (641, 10 ** 9)):
        assert len(set(share[(counts >= lo) & (counts <= hi)])) > 1
    gpu, ref = run_pair(p, s, 3)
    a = gpu.trace(0)[0]
    assert ((a & 4) == 0).sum() > 0.5 * len(a) and ((a & 4) != 0).any()
