"""The limit of the device-side waits (wait_polls): the largest value a caller may pass never runs out."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
LARGEST = 2 ** 63 - 1


def test_limit_leaves_room_for_the_kernels_factors(tmp_path):
    src, lib = tmp_path / "harness.cpp", tmp_path / "harness.so"
    src.write_text('#include "eik_host.h"\n'
                   'extern "C" long long limit(long long polls, long long preset) {'
                   ' return eikh::wait_limit(polls, preset); }\n')
    subprocess.run(["g++", "-std=c++17", "-fPIC", "-shared", "-I" + os.path.join(ROOT, "include"),
                    "-I" + os.path.join(ROOT, "paper_1811_00009_gb300", "csrc"), str(src), "-o", str(lib)], check=True)
    f = C.CDLL(str(lib)).limit
    f.restype, f.argtypes = C.c_longlong, [C.c_longlong] * 2
    preset = 1 << 22
    assert f(0, preset) == preset and f(1, preset) == 1 and f(12345, preset) == 12345
    for polls in (LARGEST, 2 ** 60, 2 ** 57):
        assert preset < f(polls, preset) <= LARGEST // 64


def test_shorter_naps_take_more_polls(tmp_path):
    """A wait with shorter naps than the 4 us the limit counts takes as many more polls, and a warp that watches its CTA's
    poller waits longer than the poller."""
    from paper_1811_00009_gb300 import build
    src, lib = tmp_path / "naps.cpp", tmp_path / "naps.so"
    src.write_text('#include "eik_internal.cuh"\n'
                   'extern "C" int unit() { return eikg::kWaitNap; }\n'
                   'extern "C" int barrier() { return eikg::kBarrierPolls * eikg::kBarrierNap; }\n'
                   'extern "C" int watch() { return eikg::kWatchPolls * eikg::kWatchNap; }\n')
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-fPIC", "-shared", "-I" + cuda, "-I" + build.CSRC, str(src), "-o", str(lib)],
                   check=True)
    L = C.CDLL(str(lib))
    assert L.unit() == 4096 and L.barrier() >= L.unit() and L.watch() >= 2 * L.barrier()


@pytest.mark.gpu
@pytest.mark.parametrize("kw", [dict(block_dim=8), dict(block_dim=16), dict(block_dim=32), dict(schedule=2, seed=3)],
                         ids=["blocks8", "blocks16", "blocks32", "random"])
def test_largest_limit_solves(kw):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1811_00009_gb300 import build
    build.build()
    import paper_1811_00009_gb300 as eik
    w = synth.workload("C2", 64)
    F = np.ascontiguousarray(w.speed().astype(np.float32))
    with eik.Solver(w.dims, w.h, F, "fp32") as S:
        S.add_sources(w.sources)
        S.solve(2 * w.h, block_dim=8)
        base = S.result().copy()
        for polls in (LARGEST, 2 ** 60 + 1):
            S.solve(2 * w.h, wait_polls=polls, **kw)
            assert np.array_equal(S.result(), base)
