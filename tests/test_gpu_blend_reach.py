"""Alpha-blending render where its block skipping can go wrong: Gaussians much
smaller than a block, needles, large and off-image ones, opacities around the
1/255 limit, images smaller than a tile and lists longer than one staging
batch. The walk's decisions are compared with the oracle through each
pixel's last contributing entry, so a wrongly skipped entry shows."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [
    # (W, H, n, smallest and largest scale, logit range)
    (40, 24, 400, 0.2, 0.6, (-1, 2)),      # far smaller than a block
    (64, 64, 300, 0.4, 30.0, (-7, -4)),    # opacities around 1/255, narrow and large ones
    (13, 9, 200, 0.5, 4.0, (-1, 4)),       # image inside one tile
    (48, 32, 2500, 1.0, 8.0, (-4, -2)),    # lists of several staging batches
]


@pytest.fixture(scope="module")
def gi():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2403_08551_gb300 as m
    m.load()
    return m


@pytest.mark.parametrize("W,H,n,lo,hi,logits", CASES)
def test_walk_matches_oracle(gi, W, H, n, lo, hi, logits):
    g = np.random.default_rng(n)
    means, _, color = synth.init_gaussians(n, W, H, n)
    means = (means * 1.2 - 0.1 * np.array([W, H])).astype(np.float32)  # some centres outside
    chol = np.stack([np.exp(g.uniform(np.log(lo), np.log(hi), n)), g.uniform(-2, 2, n) * hi / 8,
                     np.exp(g.uniform(np.log(lo), np.log(hi), n))], 1).astype(np.float32)
    logit = g.uniform(*logits, n).astype(np.float32)
    target = synth.image(W, H, n, n_blobs=5)
    p = np.concatenate([means, chol, color], 1).astype(np.float32)
    fit = gi.Fit([torch.from_numpy(target).cuda()], [torch.from_numpy(p).cuda()], tile=16, opacity="blend",
                 opacity_logits=[torch.from_numpy(logit).cuda()])
    fit.step(1)
    torch.cuda.synchronize()
    r = oracle.blend_forward_backward(means, chol, color, logit, target, 16)
    ok = ~r["ambiguous"]  # a decision within FP32 rounding of a threshold may fall either way
    assert ok.mean() > 0.9
    np.testing.assert_array_equal(fit.n_last.cpu().numpy().reshape(H, W)[ok], r["n_last"][ok])
    np.testing.assert_allclose(fit.images()[0].cpu().numpy()[ok], r["out"][ok], rtol=0,
                               atol=5e-5 * max(1.0, np.abs(r["out"]).max()))
    fit.close()
    assert gi.device_errors() == 0
