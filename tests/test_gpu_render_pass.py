"""The fused passes (gi_render_pass behind Renderer, gi_rasterize_* behind
rasterize) against the separate per-stage calls: same kernels and order, so
image, binning and gradients agree bit for bit, on both binning paths, every
tile edge, the second attempt after a short capacity guess and no Gaussians."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [
    # (W, H, n, T, scale)
    (70, 41, 300, 16, 1.0),      # count matrix, ragged image
    (200, 150, 9000, 8, 1.0),    # 475 tiles, 256-Gaussian chunks
    (61, 45, 1, 32, 1.0),
    (1100, 700, 4000, 16, 1.0),  # 3,036 tiles: radix
    (256, 256, 900, 8, 5.0),     # more than 8 pairs a Gaussian: the capacity guess is short
    (700, 420, 800, 8, 5.0),     # the same on the radix path
    (64, 32, 0, 16, 1.0),
]


@pytest.fixture(scope="module")
def gi():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2403_08551_gb300 as m
    m.load()
    return m


@pytest.mark.parametrize("W,H,n,T,scale", CASES)
def test_fused_passes_equal_the_stages(gi, W, H, n, T, scale):
    means, chol, color = synth.init_gaussians(n, W, H, n + T)
    m, l, c = (torch.from_numpy(a).cuda() for a in (means, (chol * np.float32(scale)).astype(np.float32), color))
    rec, rect, cnt = gi.project(m, l, c, W, H, T)
    b = gi.bin_tiles(rect, cnt, rec, W, H, T)
    ref = gi.render(b, W, H, T)[0]
    r = gi.Renderer(W, H, n, T, capacity=max(64, 2 * b.K))
    assert torch.equal(r(m, l, c), ref)
    assert torch.equal(r.rect, rect) and torch.equal(r.cnt, cnt) and int(r.k_dev) == b.K
    assert torch.equal(r.ids[:b.K], b.ids[:b.K]) and torch.equal(r.keys[:b.K], b.keys[:b.K])
    assert torch.equal(r.ranges, b.ranges) and torch.equal(r.pair_off, b.pair_off)
    leaf = [t.clone().requires_grad_() for t in (m, l, c)]
    out = gi.rasterize(*leaf, W, H, T)
    assert torch.equal(out.detach(), ref)
    up = torch.randn(H, W, 3, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    got = torch.autograd.grad(out, leaf, up.transpose(0, 1).contiguous().transpose(0, 1))  # not contiguous
    if n:
        want = gi.render_backward(b, rect, cnt, l, up, W, H, T)
        for x, y in zip(got, want):
            assert torch.equal(x, y)
    assert gi.device_errors() == 0


def test_rasterize_from_two_threads_and_streams(gi):
    import threading
    W, H, n, T = 200, 120, 1500, 16
    res = {}

    def work(k):
        m, l, c = (torch.from_numpy(a).cuda() for a in synth.init_gaussians(n, W, H, k))
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s):
            for _ in range(20):
                out = gi.rasterize(m, l, c, W, H, T)
            s.synchronize()
        res[k] = out

    th = [threading.Thread(target=work, args=(k,)) for k in (1, 2)]
    for t in th:
        t.start()
    for t in th:
        t.join()
    for k in (1, 2):
        m, l, c = (torch.from_numpy(a).cuda() for a in synth.init_gaussians(n, W, H, k))
        assert torch.equal(res[k], gi.rasterize(m, l, c, W, H, T))
