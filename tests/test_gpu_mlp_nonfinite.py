"""The schedule network's gradient with values that are not finite: a sample's reach only what depends on that sample, and
a block's unused places (fewer samples than the block holds) contribute nothing, whatever the weights are.

W3's and b3's gradient of an action sums over the samples that took it, so those of other actions stay what they are
without the bad sample; 2e-3 of the largest entry is twice the gradient's bar of test_gpu_mlp.py."""
import numpy as np
import pytest

import synth
from oracle import mlp

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


def gradient(eik, w, X, act, tgt):
    import torch
    wd, Xd, ad, td = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (w, X, act, tgt)]
    g = torch.empty(mlp.n_params(), device="cuda")
    loss = torch.empty(1, device="cuda")
    work = torch.empty(eik.eik_mlp_work_floats(len(X)), device="cuda")
    eik.eik_mlp_grad(wd, Xd, ad, td, g, loss, work)
    torch.cuda.synchronize()
    return g.cpu().numpy()


def data(B):
    w = (synth.normal(21, 1, mlp.n_params()) * 0.3).astype(np.float32)
    X = synth.normal(21 + B, 2, B * mlp.D_IN).reshape(B, mlp.D_IN).astype(np.float32)
    act = (synth.uniform(21 + B, 3, B) * mlp.A).astype(np.int32)
    tgt = synth.normal(21 + B, 4, B).astype(np.float32)
    return w, X, act, tgt


OFF_W3 = mlp.n_params() - mlp.A * 33                    # W3 (A x 32), then b3 (A)
OFF_B3 = mlp.n_params() - mlp.A


@pytest.mark.parametrize("B", [5, 128, 300])
@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_a_bad_sample_stays_with_its_action(eik, B, value):
    w, X, act, tgt = data(B)
    bad = B // 2
    act[bad] = 3
    X[bad, 4] = value
    w[4] = 0.0                                          # (inf times this weight: a hidden value is NaN)
    g = gradient(eik, w, X, act, tgt)
    keep = np.arange(B) != bad
    _, ref = mlp.grad(w.astype(np.float64), X[keep].astype(np.float64), act[keep], tgt[keep].astype(np.float64))
    ref = ref * (keep.sum() / B)                        # (the loss is a mean over B)
    top = np.max(np.abs(ref))
    others = [a for a in range(mlp.A) if a != 3]
    for a in others:
        assert np.all(np.abs(g[OFF_W3 + 32 * a:OFF_W3 + 32 * (a + 1)] - ref[OFF_W3 + 32 * a:OFF_W3 + 32 * (a + 1)]) <= 2e-3 * top)
        assert abs(g[OFF_B3 + a] - ref[OFF_B3 + a]) <= 2e-3 * top
    assert np.all(np.isnan(g[OFF_W3 + 96:OFF_W3 + 128]))


@pytest.mark.parametrize("B", [1, 129])
def test_unused_places_with_an_infinite_weight(eik, B):
    """An action that no sample took has infinite weights: the gradient of all others is what it is without it."""
    w, X, act, tgt = data(B)
    act[act == 0] = 1
    base = gradient(eik, w, X, act, tgt)
    w[OFF_W3:OFF_W3 + 32] = np.inf
    g = gradient(eik, w, X, act, tgt)
    assert np.all(np.isfinite(base)) and np.array_equal(g, base)
