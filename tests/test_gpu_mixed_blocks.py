"""Schedules that mix 8^3 and 16^3 restarts in channels one node wide, where the front passes from block to block through
a single node: a node lowered above the bound in a 16^3 restart, on a face between two bricks of the group, has to reach
the brick across that face when the next restarts have 8^3 blocks (nothing else does, in a channel).

Bars: finite where the FP64 oracle is; equal to the fixed 8^3 schedule bit for bit; and, with one root rounded to nearest
per node of the channel (N nodes) and h/F rounded once, within (N + 2) half last places of the largest psi (FP64: four
last places a node, since the oracle's own roots are rounded too).
"""
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


def serpentine(nx, ny, nz):
    """Open nodes of a channel one node wide: along x in every second row, the rows joined at alternating ends, the
    layers (every second z) joined where one ends and the next begins."""
    m = np.zeros((nz, ny, nx), bool)
    path = []
    fwd = True
    for z in range(0, nz, 2):
        rows = list(range(0, ny, 2))
        if (z // 2) % 2:
            rows.reverse()
        for q, y in enumerate(rows):
            xs = range(nx) if fwd else range(nx - 1, -1, -1)
            path += [(x, y, z) for x in xs]
            x_end = nx - 1 if fwd else 0
            fwd = not fwd
            if q + 1 < len(rows):
                path.append((x_end, (y + rows[q + 1]) // 2, z))
            elif z + 2 < nz:
                path.append((x_end, y, z + 1))
    for x, y, z in path:
        m[z, y, x] = True
    return m, len(path)


CHANNELS = {"x": (1024, 1, 1), "y": (1, 700, 1), "z": (1, 1, 1024), "serpentine": (64, 33, 5)}


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("name", list(CHANNELS))
def test_channels(eik, orc, name, precision):
    dims = CHANNELS[name]
    h = synth.grid_h(dims)
    open_, n = serpentine(*dims)
    rough = 10.0 ** (synth.uniform(31, 4, open_.size).reshape(open_.shape) - 0.5)
    for speeds in (np.ones(open_.shape), rough):
        F = synth.round_to(np.where(open_, speeds, 0.0), precision)
        src = [[0.0, 0.0, 0.0]]
        ref = orc.fmm(F, h, src)
        fin = np.isfinite(ref)
        assert np.array_equal(fin, open_)
        bar = (n + 2) * (2.0 ** -24 if precision == "fp32" else 2.0 ** -50) * ref[fin].max()
        with eik.Solver(dims, h, np.ascontiguousarray(F.astype(np.float32 if precision == "fp32" else np.float64)),
                        precision) as S:
            S.add_sources(src)
            S.solve(2.0 * h, block_dim=8)
            base = S.result().copy()
            assert np.array_equal(np.isfinite(base), fin)
            assert np.max(np.abs(base[fin].astype(np.float64) - ref[fin])) <= bar
            runs = [dict(schedule=eik.EIK_SCHED_RANDOM, seed=s, block_dim=b) for s in range(8) for b in (8, 16)]
            runs.append(dict(schedule=eik.EIK_SCHED_LEARNED))
            for kw in runs:
                S.solve(2.0 * h, **kw)
                assert np.array_equal(S.result(), base), kw
