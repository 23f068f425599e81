"""The region rule of concurrent moves with centres uniform in a dilute box. There A_w = A0 lam /
sqrt(nbar) exceeds A0 lam (mean support nbar below one bead), so a move can shift beads further than
A0 lam / 4: every move that ran concurrently must have its whole influence ball, lam + A_w / 4 + the
interaction reach about its centre, in fine cells of its own region (restated here from the counter
stream). On the GPU every decision, position and counter against the oracle."""
import math

import numpy as np
import pytest

import oracle as O
from paper_1611_09160_gb300 import inputs as I
from paper_1611_09160_gb300 import wmcd

K_BUNI = 18


def case(eps, precision=wmcd.FP64, n=600, phi=1e-3, K=2, **kw):
    s = I.free_spheres(n, phi, seed=9)
    p = wmcd.default_params(s.n_beads, s.box_L, seed=77, precision=precision, centring=wmcd.CENTRE_UNIFORM,
                            bond_type=wmcd.BOND_NONE, wca_eps=eps, A0=1.0, colour_K=K, **kw)
    g = 8 * K // 2
    p["grid_layer"] = [g, g // 2 // K * K] + [0] * 14
    return s, p


@pytest.mark.parametrize("eps, K", [(0.0, 2), (1.0, 2), (0.0, 3)])
def test_concurrent_moves_stay_in_their_region(eps, K):
    s, p = case(eps, K=K)
    L, Gf, A0, N = s.box_L, p["grid_f"], p["A0"], s.n_beads
    reach = (2.0 ** (1.0 / 6.0) * p["wca_sigma"] if eps else 0.0) + 1e-6
    key = [p["seed"] & 0xffffffff, (p["seed"] >> 32) ^ p["sim_id"]]
    ref = O.Oracle(p, s.pos, s.chain_len)
    ran = wide = 0
    for sweep in range(3):
        ref.sweep(1)
        for l in range(2):
            G = p["grid_layer"][l]
            out, n = ref.trace_layer(l)
            lam = ref.trace_lam(l)
            for j in np.nonzero(((out & 3) != 0) & ((out & 4) == 0))[0]:
                w = O.philox([j, sweep, (K_BUNI << 24) | (l << 16), 0], key)
                nbar = N * (4.0 * math.pi / 3.0) * lam[j] ** 3 / L ** 3
                disp = 0.25 * A0 * lam[j] / math.sqrt(nbar)
                ran += 1
                wide += nbar < 1.0
                for a in range(3):
                    b = L * (float(w[a]) / 2.0 ** 32)
                    c = min(int(b * G / L), G - 1)
                    lo = -((-(2 * c - (K - 1)) * Gf) // (2 * G))
                    hi = ((2 * c + 2 + (K - 1)) * Gf) // (2 * G) - 1
                    R = (lam[j] + disp + reach) * (1.0 - 1e-12)
                    t0, t1 = math.floor((b - R) * Gf / L), math.floor((b + R) * Gf / L)
                    assert any(t0 + k >= lo and t1 + k <= hi for k in (-Gf, 0, Gf)), (l, j, a, b, lam[j], R, lo, hi)
    assert ran > 100 and wide > 50


@pytest.mark.gpu
@pytest.mark.parametrize("eps, K, level2", [(0.0, 2, 0), (1.0, 2, 0), (1.0, 2, 1), (0.0, 3, 0)])
@pytest.mark.parametrize("precision", [wmcd.FP64, wmcd.MIXED])
def test_dilute_uniform_centres_against_the_oracle(eps, K, level2, precision):
    from test_gpu_parity import run_pair
    wmcd.build()
    wmcd.load()
    s, p = case(eps, precision, K=K, level2=level2)
    gpu, ref = run_pair(p, s, 10)
    out, n = gpu.trace(0)
    assert ((out & 4) == 0).any() and (n > 0).any()


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [wmcd.FP64, wmcd.MIXED])
def test_dense_regions_in_a_dilute_box_against_the_oracle(precision):
    """All beads in one octant: supports of many beads moved by the amplitude of the mean one, in blocks
    of a queue each and (two cells per axis, every region beyond staging) by groups of blocks."""
    from test_gpu_parity import run_pair
    wmcd.build()
    wmcd.load()
    t = I.free_spheres(6000, 0.02, seed=4)
    L = 2.0 * t.box_L
    for grid in (4, 2):
        p = wmcd.default_params(t.n_beads, L, seed=5, precision=precision, centring=wmcd.CENTRE_UNIFORM,
                                bond_type=wmcd.BOND_NONE, A0=0.7)
        p["grid_layer"] = [grid] + [0] * 15
        run_pair(p, I.System(t.pos, t.chain_len, L), 1)
