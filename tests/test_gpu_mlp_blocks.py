"""The schedule network's kernels at the edges of their blocks (64 samples a block forward, 128 a block in the
gradient, eight partial sums a parameter): against the FP64 reference within the bars of test_gpu_mlp.py
(outputs 1e-4 relative + 1e-5, loss 1e-4 relative, gradient 1e-3 of its largest entry)."""
import numpy as np
import pytest

import synth
from oracle import mlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 63, 65, 127, 128, 129, 1025, 9001])
def test_sample_counts(B):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1811_00009_gb300 import build
    build.build()
    import paper_1811_00009_gb300 as eik
    w = (synth.normal(21, 1, mlp.n_params()) * 0.3).astype(np.float32)
    X = synth.normal(21 + B, 2, B * mlp.D_IN).reshape(B, mlp.D_IN).astype(np.float32)
    act = (synth.uniform(21 + B, 3, B) * mlp.A).astype(np.int32)
    tgt = synth.normal(21 + B, 4, B).astype(np.float32)
    wd, Xd, ad, td = [torch.from_numpy(a).cuda() for a in (w, X, act, tgt)]
    Y = torch.empty((B, mlp.A), device="cuda")
    g = torch.empty(mlp.n_params(), device="cuda")
    loss = torch.empty(1, device="cuda")
    work = torch.empty(eik.eik_mlp_work_floats(B), device="cuda")
    eik.eik_mlp_forward(wd, Xd, Y)
    eik.eik_mlp_grad(wd, Xd, ad, td, g, loss, work)
    torch.cuda.synchronize()
    ref, _, _ = mlp.forward(w.astype(np.float64), X.astype(np.float64))
    np.testing.assert_allclose(Y.cpu().numpy(), ref, rtol=1e-4, atol=1e-5)
    l_ref, g_ref = mlp.grad(w.astype(np.float64), X.astype(np.float64), act, tgt.astype(np.float64))
    assert abs(loss.item() - l_ref) <= 1e-4 * abs(l_ref)
    assert np.max(np.abs(g.cpu().numpy() - g_ref)) <= 1e-3 * np.max(np.abs(g_ref))
