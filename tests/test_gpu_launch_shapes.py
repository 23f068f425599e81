"""Launch shapes of a lone simulation: with a serial block of 32 or 128 threads no launch waits until every
SM is free, neither the serial phases nor the regions beyond staging. A kernel that keeps one SM's shared
memory for a bounded time stands for the other work of a program; the results are those of the default."""
import ctypes
import subprocess
import time

import numpy as np
import pytest

from paper_1611_09160_gb300 import inputs as I
from paper_1611_09160_gb300 import wmcd

pytestmark = pytest.mark.gpu

HOLD_S = 1.0
HOLD = r"""
#include <cuda_runtime.h>
__global__ void hold(long long ns) {            // one thread, until the timer has run ns (or 2^26 reads of it)
    extern __shared__ char keep[];
    long long t0, t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
    for (int i = 0; i < (1 << 26); i++) {
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
        if (t - t0 >= ns) break;
    }
    keep[0] = (char)t;
}
extern "C" int start_hold(long long ns, void* stream) {
    cudaFuncSetAttribute(hold, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
    hold<<<1, 1, 100 * 1024, (cudaStream_t)stream>>>(ns);
    return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module", autouse=True)
def built():
    wmcd.build()
    wmcd.load()


@pytest.fixture(scope="module")
def hold(tmp_path_factory):
    d = tmp_path_factory.mktemp("hold")
    src, so = d / "hold.cu", d / "libhold.so"
    src.write_text(HOLD)
    nvcc = "/usr/local/cuda/bin/nvcc"
    subprocess.check_call([nvcc] + wmcd.ARCH_FLAGS + ["-O2", "-shared", "-Xcompiler", "-fPIC", "-o", str(so), str(src)])
    f = ctypes.CDLL(str(so)).start_hold
    f.argtypes = [ctypes.c_longlong, ctypes.c_void_p]
    return f


@pytest.mark.parametrize("precision", [wmcd.FP64, wmcd.MIXED])
@pytest.mark.parametrize("threads", [32, 128])
def test_one_block_form_runs_beside_other_work(threads, precision, hold):
    import torch
    s = I.make_system([20] * 1000, 0, I.box_for_volume_fraction(20000, 0.2), seed=41)
    p = wmcd.default_params(s.n_beads, s.box_L, seed=19, precision=precision, n_cap=12, lambda_max=4.0)
    p["grid_layer"] = [4] + [0] * 15                   # eight regions a phase, about 2,500 beads each
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    runs = []
    for block in (None, (2, threads)):
        sim = wmcd.Simulation(p, s.pos, s.chain_len, stream=mine)
        if block:
            sim.set_block(*block)
        t = time.perf_counter()
        sim.sweep(1, stream=mine)                      # the first sweep alone, the second beside the kernel
        mine.synchronize()
        alone = time.perf_counter() - t
        if block:
            t = time.perf_counter()
            assert hold(int(1e9 * HOLD_S), other.cuda_stream) == 0
        sim.sweep(1, stream=mine)
        mine.synchronize()
        if block:
            beside = time.perf_counter() - t
            other.synchronize()
            assert alone < 0.5 * HOLD_S and beside < 0.8 * HOLD_S, (alone, beside)
        runs.append((sim.positions(stream=mine), sim.trace(0, stream=mine)))
        sim.close()
    (x, t), (y, u) = runs
    assert np.array_equal(x, y) and np.array_equal(t[0], u[0]) and np.array_equal(t[1], u[1])
