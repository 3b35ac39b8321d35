"""Count-matrix binning where its dispatch changes: the chunk size (128
Gaussians up to 8,192, then 256) and the column sums taken by the placement
itself (up to 8,192 counts) or by their own kernel. Integer work, compared
with the oracle bit for bit, standalone and inside a fit (whose projection
writes the counts)."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [
    # (W, H, n, T)
    (256, 256, 4096, 16),   # 32 chunks x 256 tiles = 8,192 counts: summed by the placement
    (256, 256, 4097, 16),   # 33 chunks: by the column scan
    (256, 256, 8192, 16),   # last size with 128-Gaussian chunks
    (256, 256, 8193, 16),   # 256-Gaussian chunks, a chunk of one
    (70, 40, 8500, 32),     # 34 chunks x 6 tiles: placement sums, many pairs a tile
    (48, 33, 1, 16),        # one Gaussian
]


@pytest.fixture(scope="module")
def gi():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2403_08551_gb300 as m
    m.load()
    return m


@pytest.mark.parametrize("W,H,n,T", CASES)
def test_binning_matches_oracle_around_the_dispatch(gi, W, H, n, T):
    means, chol, color = synth.init_gaussians(n, W, H, n)
    rect_ref, cnt_ref = oracle.rect_rule(means, chol, color, W, H, T)
    ids_ref, ranges_ref, off_ref = oracle.bin_tiles(rect_ref, cnt_ref, W, H, T)
    m, l, c = (torch.from_numpy(a).cuda() for a in (means, chol, color))
    rec, rect, cnt = gi.project(m, l, c, W, H, T)
    b = gi.bin_tiles(rect, cnt, rec, W, H, T)
    K = ids_ref.shape[0]
    assert b.K == K
    np.testing.assert_array_equal(b.ids[:K].cpu().numpy().astype(np.uint32), ids_ref)
    np.testing.assert_array_equal(b.ranges.cpu().numpy(), ranges_ref)
    np.testing.assert_array_equal(b.pair_off.cpu().numpy(), off_ref)
    assert torch.equal(b.rec_binned[:K], rec[b.ids[:K].long()])
    p = torch.from_numpy(np.concatenate([means, chol, color], axis=1)).cuda()
    fit = gi.Fit([torch.rand(H, W, 3, device="cuda")], [p], tile=T)
    fit.step(1)
    f = fit.binning()
    np.testing.assert_array_equal(f["ids"].cpu().numpy().astype(np.uint32), ids_ref)
    np.testing.assert_array_equal(f["ranges"].cpu().numpy(), ranges_ref)
    np.testing.assert_array_equal(f["pair_off"].cpu().numpy(), off_ref)
    fit.close()
    assert gi.device_errors() == 0
