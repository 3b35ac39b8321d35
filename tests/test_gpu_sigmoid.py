"""The double-float sigmoid of the formation (opacities, App. C.1 positions)
against the oracle's FP64 values: a value that its relative error of at most
2^-42.8 could round either way is taken in FP64, so the rounded results are
the oracle's."""
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


def params(n, W, H, seed):
    return np.concatenate(synth.init_gaussians(n, W, H, seed), axis=1).astype(np.float32)


@pytest.mark.parametrize("lo,hi", [(-4, 4), (-30, 30), (-110, -80)])
def test_opacity_is_rounded_like_fp64(gi, lo, hi):
    n, W, H = 200000, 64, 64
    g = np.random.default_rng(7)
    logit = g.uniform(lo, hi, n).astype(np.float32)
    logit[:8] = [0.0, -0.0, 1e-30, -1e-30, 88.0, -88.0, 1000.0, -1000.0]
    fit = gi.Fit([torch.zeros(H, W, 3, device="cuda")], [torch.from_numpy(params(n, W, H, 1)).cuda()], opacity="separate",
                 opacity_logits=[torch.from_numpy(logit).cuda()])
    fit.render()
    torch.cuda.synchronize()
    o, ref = fit.opacity.cpu().numpy(), oracle.sigmoid_opacity(logit)
    fit.close()
    ulps = np.abs(o.view(np.int32).astype(np.int64) - ref.view(np.int32).astype(np.int64))
    assert ulps.max() == 0
    np.testing.assert_array_equal(o[:8], ref[:8])


@pytest.mark.parametrize("T", [8, 16])
def test_raw_positions_give_the_oracles_rectangles(gi, T):
    n, W, H = 100000, 517, 389
    p = params(n, W, H, 2)
    g = np.random.default_rng(3)
    p[:, 0:2] = np.arctanh(g.uniform(-0.9999, 0.9999, (n, 2)))
    p[: n // 4, 0:2] = g.uniform(-12, 12, (n // 4, 2))  # far outside the usual range: at the borders
    p[0, 0:2], p[1, 0:2], p[2, 0:2] = (np.inf, 0), (-np.inf, 0), (np.nan, 0)
    fit = gi.Fit([torch.zeros(H, W, 3, device="cuda")], [torch.from_numpy(p).cuda()], tile=T, param_mode="paper")
    fit.render()
    b = fit.binning()
    means, chol, _ = oracle.paper_formation(p[:, 0:2], p[:, 2:5], W, H)
    rect, cnt = oracle.rect_rule(means, chol, p[:, 5:8], W, H, T)
    np.testing.assert_array_equal(b["rect"].cpu().numpy(), rect)
    np.testing.assert_array_equal(b["cnt"].cpu().numpy(), cnt)
    fit.close()
