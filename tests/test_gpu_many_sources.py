"""Hundreds of on-node sources at brick corners, far apart: each activates four bricks in four 16^3 groups, the most
entries a source brings to the first work lists."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_spread_corner_sources(orc, precision):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1811_00009_gb300 import build
    build.build()
    import paper_1811_00009_gb300 as eik
    dims = (185, 190, 187)
    h = synth.grid_h(dims)
    F = synth.round_to(0.5 + synth.uniform(17, 1, int(np.prod(dims))).reshape(dims[::-1]), precision)
    src = h * (32.0 * np.stack(np.meshgrid(*[np.arange(6)] * 3, indexing="ij"), -1).reshape(-1, 3) + 16.0)
    with eik.Solver(dims, h, np.ascontiguousarray(F.astype(np.float32 if precision == "fp32" else np.float64)),
                    precision) as S:
        S.add_sources(src)
        S.solve(2.0 * h, block_dim=8)
        base = S.result().copy()
        for kw in (dict(block_dim=16), dict(schedule=eik.EIK_SCHED_LEARNED),
                   dict(schedule=eik.EIK_SCHED_RANDOM, seed=2, block_dim=16)):
            S.solve(2.0 * h, **kw)
            assert np.array_equal(S.result(), base), kw
    ref = orc.fmm(F, h, src)
    if precision == "fp32":
        assert np.max(np.abs(base.astype(np.float64) - ref)) <= 1e-5 * ref.max()
    else:
        assert np.all(np.abs(base - ref) <= 1e-12 * ref)
