"""32^3 blocks where a wave has more nodes than its list holds (16384): with a source on every seventh node, all others next
to one, the first wave's neighbours are most of the block.  What does not fit waits, marked, for a later wave.

Same bits as the 8^3 blocks, and within 1e-5 of the largest psi of the FP64 oracle (the bar of test_gpu_block32.py)."""
import math

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

LIST = 16384


@pytest.mark.parametrize("dims", [(32, 32, 32), (45, 37, 64)])
@pytest.mark.parametrize("rough", [False, True])
def test_a_wave_of_most_of_a_block(orc, dims, rough):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1811_00009_gb300 import build
    build.build()
    import paper_1811_00009_gb300 as eik
    h = synth.grid_h(dims)
    n = int(np.prod(dims))
    z, y, x = np.meshgrid(*[np.arange(d) for d in dims[::-1]], indexing="ij")
    on = (x + 2 * y + 3 * z) % 7 == 0
    near = np.zeros_like(on)
    for axis in range(3):
        for step in (1, -1):
            near[:] |= np.roll(on, step, axis)
    assert np.count_nonzero((near & ~on)[:32, :32, :32]) > LIST
    u = synth.uniform(611, 2, 2 * n)
    F = np.ones(n) if not rough else np.where(u[n:] < 0.05, 0.0, 10.0 ** (2.0 * u[:n] - 1.0))
    F = F.reshape(dims[::-1]).astype(np.float32)
    src = h * np.stack([x[on], y[on], z[on]], -1).astype(np.float64)
    with eik.Solver(dims, h, np.ascontiguousarray(F), "fp32") as S:
        S.add_sources(src)
        S.solve(2.0 * h, block_dim=8)
        base = S.result().copy()
        for stride, window in ((2.0, 2.0), (math.inf, 1e6), (0.5, 1e-3)):
            S.solve(stride * h, block_dim=32, window=window)
            assert np.array_equal(S.result(), base), (stride, window)
    ref = orc.fmm(F.astype(np.float64), h, src)
    fin = np.isfinite(ref)
    assert np.array_equal(np.isfinite(base), fin)
    assert np.max(np.abs(base[fin].astype(np.float64) - ref[fin])) <= 1e-5 * ref[fin].max()
