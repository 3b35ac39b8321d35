"""The radix binning's sort where it changes the number of keys a thread takes:
one wave is 152 blocks of 512 threads, so 4, 8, 12 and 16 keys a thread hold
311,296, 622,592, 933,888 and 1,245,184 keys; beyond, 12 or 16 by the waves.
Every Gaussian covers one tile, so the pair count is exact and the order is a
stable sort by tile."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
WAVE = 152 * 512


@pytest.fixture(scope="module")
def gi():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2403_08551_gb300 as m
    m.load()
    return m


@pytest.mark.parametrize("spread", [1, 4])
@pytest.mark.parametrize("n", [1, 2049, 4 * WAVE, 4 * WAVE + 1, 8 * WAVE, 8 * WAVE + 1, 12 * WAVE, 12 * WAVE + 1,
                               16 * WAVE + 1, 24 * WAVE + 1, 36 * WAVE - 1])
def test_sort_is_stable_at_every_block_size(gi, n, spread):
    T, tw, th = 16, 64, 48  # 3,072 tiles: above the count matrix
    g = np.random.default_rng(n)
    t = g.integers(0, tw * th // spread, n)  # spread 4: a quarter of the tiles, so longer runs
    x, y = t % tw, t // tw
    rect = np.stack([x, y, x + 1, y + 1], 1).astype(np.int32)
    b = gi.bin_tiles(torch.from_numpy(rect).cuda(), torch.ones(n, dtype=torch.int32, device="cuda"), None, tw * T, th * T,
                     T, capacity=n)
    order = np.argsort(t, kind="stable")
    assert b.K == n
    np.testing.assert_array_equal(b.ids.cpu().numpy(), order)
    np.testing.assert_array_equal(b.keys.cpu().numpy(), t[order])
    start = np.searchsorted(t[order], np.arange(tw * th + 1))
    full = np.diff(start) > 0
    np.testing.assert_array_equal(b.ranges.cpu().numpy()[full], np.stack([start[:-1], start[1:]], 1)[full])
    assert gi.device_errors() == 0
