"""The queue marches of the 8^3 and 16^3 blocks (eik_march8.cuh, eik_march16.cuh) where they can go wrong: rough speeds (many stages in a
march, corrections of accepted values), barriers, sources on block faces, grids of one node to a few blocks with
ragged edges, and windows and strides from one node a stage to the whole block at once.

Every variant must give the discrete solution of the FP64 oracle within the precision bars of the parity tests
(FP64: relative 1e-12; FP32: 1e-5 of the largest psi, the accumulated rounding of one root per node along a
characteristic) and must equal the first variant bit for bit (the update is monotone, so the order of the work
does not matter).
"""
import math

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eik():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1811_00009_gb300 import build
    build.build()
    import paper_1811_00009_gb300 as E
    return E


VARIANTS = [dict(stride=2.0), dict(stride=0.3), dict(stride=1.0, window=1e-3), dict(stride=5.0, window=0.5),
            dict(stride=math.inf), dict(stride=math.inf, window=50.0), dict(stride=3.0, fallback_tau=1.0)]


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("dims", [(1, 1, 1), (8, 8, 8), (9, 7, 8), (17, 8, 25), (31, 33, 16)])
def test_rough_speeds_and_barriers(eik, orc, dims, precision):
    n = int(np.prod(dims))
    h = synth.grid_h(dims)
    u = synth.uniform(91 + n, 2, 2 * n)
    F = (10.0 ** (2.0 * u[:n] - 1.0)).reshape(dims[::-1])             # 0.1 .. 10
    F[(u[n:] < 0.12).reshape(dims[::-1])] = 0.0
    F[0, 0, 0] = 1.0
    F = synth.round_to(F, precision)
    src = [[0.0, 0.0, 0.0]]
    if min(dims) > 8:
        src += [[8 * h, 8 * h, 7.5 * h], [(dims[0] - 1) * h, 0.3 * h, 9 * h]]
    ref = orc.fmm(F, h, src)
    fin = np.isfinite(ref)
    dt = np.float32 if precision == "fp32" else np.float64
    base = None
    with eik.Solver(dims, h, np.ascontiguousarray(F.astype(dt)), precision) as S:
        S.add_sources(src)
        for v in VARIANTS:
            kw = dict(v)
            stride = kw.pop("stride") * h
            for edge in (8, 16):
                S.solve(stride, block_dim=edge, **kw)
                psi = S.result()
                assert np.array_equal(np.isfinite(psi), fin), (v, edge)
                if precision == "fp64":
                    assert np.all(np.abs(psi[fin] - ref[fin]) <= 1e-12 * ref[fin]), (v, edge)
                else:
                    assert np.max(np.abs(psi[fin].astype(np.float64) - ref[fin])) <= 1e-5 * ref[fin].max(), (v, edge)
                base = psi.copy() if base is None else base
                assert np.array_equal(psi, base), (v, edge)


def test_block32_lists_overflow_and_mixed_blocks(eik, orc):
    """32^3 blocks where a wave's nodes are many (one stage spans the whole block: infinite stride, wide window)
    and where they are few, rough speeds, ragged grid of 2x2x2 blocks: the 8^3 result bit for bit."""
    dims = (45, 37, 52)
    h = synth.grid_h(dims)
    u = synth.uniform(577, 2, 2 * int(np.prod(dims)))
    n = int(np.prod(dims))
    F = (10.0 ** (2.0 * u[:n] - 1.0)).reshape(dims[::-1])
    F[(u[n:] < 0.05).reshape(dims[::-1])] = 0.0
    F[0, 0, 0] = F[31, 31, 31] = 1.0
    F = F.astype(np.float32)
    with eik.Solver(dims, h, np.ascontiguousarray(F), "fp32") as S:
        S.add_sources([[0.0, 0.0, 0.0], [31 * h, 31 * h, 31 * h]])
        S.solve(2 * h, block_dim=8)
        base = S.result()
        ref = orc.fmm(F.astype(np.float64), h, [[0.0, 0.0, 0.0], [31 * h, 31 * h, 31 * h]])
        fin = np.isfinite(ref)
        assert np.array_equal(np.isfinite(base), fin)
        assert np.max(np.abs(base[fin].astype(np.float64) - ref[fin])) <= 1e-5 * ref[fin].max()
        for stride, window in ((2.0, 2.0), (4.0, 4.0), (1.0, 1e-3), (math.inf, 1e6), (math.inf, 2.0)):
            S.solve(stride * h, block_dim=32, window=window)
            assert np.array_equal(S.result(), base), (stride, window)


@pytest.mark.parametrize("dims", [(184, 184, 184), (192, 189, 184), (448, 432, 408)])
def test_launch_sizes(eik, dims):
    """The 8^3 loop as built for one, two and three blocks of threads an SM (grids on both sides of the first line and
    above the second), a fixed and a random schedule (8^3 and 16^3 restarts in turn): the 16^3 loop's result bit for bit."""
    import torch
    h = synth.grid_h(dims)
    g = torch.Generator(device="cuda").manual_seed(dims[0])
    F = (10.0 ** (torch.rand(dims[::-1], generator=g, device="cuda") - 0.5)).float()
    with eik.Solver(dims, h, F, "fp32") as S:
        S.add_sources([[0.0, 0.0, 0.0], [0.5 * dims[0] * h, 0.7 * dims[1] * h, 0.4 * dims[2] * h]])
        S.solve(2.0 * h, block_dim=16)
        base = S.result().copy()
        assert np.all(np.isfinite(base))
        for kw in (dict(block_dim=8), dict(schedule=eik.EIK_SCHED_RANDOM, seed=5)):
            S.solve(2.0 * h, **kw)
            assert np.array_equal(S.result(), base), kw
