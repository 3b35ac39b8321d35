"""Alpha-blending gradients when target pixels are not finite: a pixel adds
nothing to a Gaussian that it skips (alpha < 1/255), so Gaussians that no such
pixel sees keep the gradients of a finite target bit for bit."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gi():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2403_08551_gb300 as m
    m.load()
    return m


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_unseen_gaussians_keep_finite_gradients(gi, value):
    W, H, n = 48, 32, 400
    means, _, color = synth.init_gaussians(n, W, H, 5)
    g = np.random.default_rng(6)
    chol = np.stack([g.uniform(0.5, 2.0, n), g.uniform(-0.5, 0.5, n), g.uniform(0.5, 2.0, n)], 1).astype(np.float32)
    logit = g.uniform(-2, 2, n).astype(np.float32)
    p = np.concatenate([means, chol, color], 1).astype(np.float32)
    target = synth.image(W, H, 5, n_blobs=5).astype(np.float32)
    bad = [(5, 7), (19, 20), (0, 47), (31, 16)]  # (row, column)

    def grads(t):
        fit = gi.Fit([torch.from_numpy(t).cuda()], [torch.from_numpy(p).cuda()], tile=16, opacity="blend",
                     opacity_logits=[torch.from_numpy(logit).cuda()])
        fit.step(1)
        torch.cuda.synchronize()
        out = fit.grads.cpu().numpy().copy(), fit.opacity_grad.cpu().numpy().copy()
        fit.close()
        return out

    t = target.copy()
    seen = np.zeros(n, bool)
    o = oracle.sigmoid_opacity(logit).astype(np.float64)
    l1, l2, l3 = chol.astype(np.float64).T
    for y, x in bad:
        t[y, x] = value
        dx, dy = x + 0.5 - means[:, 0].astype(np.float64), y + 0.5 - means[:, 1].astype(np.float64)
        u = dx / l1                       # |L^-1 d|^2 / 2 with Sigma = L L^T
        v = (dy - l2 * u) / l3
        seen |= o * np.exp(-0.5 * (u * u + v * v)) > 0.9 / 255.0
    assert 0 < seen.sum() < n // 2
    (ga, oa), (gb, ob) = grads(target), grads(t)
    assert np.isfinite(ga).all() and np.isfinite(oa).all()
    np.testing.assert_array_equal(gb[~seen], ga[~seen])
    np.testing.assert_array_equal(ob[~seen], oa[~seen])
    assert not np.isfinite(gb[seen]).all()
