"""Host rules for the launch shapes of a colour phase (plain arithmetic, compiled here): the queues that
fill the GPU are those of all simulations of the launch."""
import ctypes
import os
import subprocess

import pytest

from paper_1611_09160_gb300 import autotune

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1611_09160_gb300", "csrc")
SMS = 152


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("shapes")
    (d / "t.cpp").write_text(
        '#include "wmcd_shapes.h"\n'
        'extern "C" int slots(int nq, int S, long long n, int sm) { return wmcd::phase_shape(nq, S, n, sm).slots; }\n'
        'extern "C" int wide(int nq, int S, long long n, int sm) { return wmcd::phase_shape(nq, S, n, sm).wide; }\n'
        'extern "C" int light(int w) { return wmcd::light_queues(w); }\n')
    so = str(d / "t.so")
    subprocess.check_call(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", so, str(d / "t.cpp")])
    lib = ctypes.CDLL(so)
    for f in (lib.slots, lib.wide):
        f.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_longlong, ctypes.c_int]
    return lib


def test_lone_simulations(rules):
    # 16k dilute beads; a dense box of eight regions; FENE chains; the large suspension's finest layer
    assert [rules.slots(n, 1, N, SMS) for n, N in ((512, 16384), (8, 65536), (3375, 20000), (58 ** 3, 5024000))] == [4, 4, 4, 24]
    assert [rules.wide(n, 1, N, SMS) for n, N in ((512, 16384), (8, 65536), (1000, 10 ** 6), (3375, 20000))] == [1, 1, 0, 0]


@pytest.mark.parametrize("nq, N", [(125, 4096), (27, 4096), (512, 16384), (1, 100)])
def test_a_batch_counts_the_queues_of_all_members(rules, nq, N):
    for S in (1, 2, 7, 64, 1024, 65535):
        assert rules.slots(nq, S, N, SMS) == (4 if nq * S <= 32 * SMS else 24)
        if nq * S > 16 * SMS:
            assert rules.wide(nq, S, N, SMS) == 0
    assert rules.wide(nq, 2, N, SMS) == rules.wide(nq, 1, N, SMS)


def test_the_tuner_times_no_shape_twice(rules):
    shapes = [(rules.light(w), t) for w, t in autotune.LAUNCH_CANDIDATES]
    assert len(set(shapes)) == len(shapes)
    assert {rules.light(w) for w in (1, 2, 3, 4)} == {q for q, _ in shapes}
