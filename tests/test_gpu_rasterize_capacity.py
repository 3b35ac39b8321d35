"""gi_rasterize_forward around the capacity that the pairs need: one pair short
it reports the count and renders nothing (a list cut off is not worth the
render's time), at the exact count it renders as the separate stages do."""
import ctypes

import pytest

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


@pytest.mark.parametrize("W,H,n,T", [(256, 256, 900, 8), (700, 420, 800, 8), (1100, 700, 4000, 16), (70, 41, 1, 32)])
def test_a_short_capacity_renders_nothing(gi, W, H, n, T):
    from paper_2403_08551_gb300 import _lib as L
    lib = L.load()
    m, l, c = (torch.from_numpy(a).cuda() for a in synth.init_gaussians(n, W, H, n + T))
    rec, rect, cnt = gi.project(m, l, c, W, H, T)
    b = gi.bin_tiles(rect, cnt, rec, W, H, T)
    ref = gi.render(b, W, H, T)[0]
    img = L.GIImage(W, H, T)
    for cap, short in ((b.K - 1, True), (b.K, False)):
        if cap < 1:
            continue
        fwd, bwd, pairs = ctypes.c_size_t(0), ctypes.c_size_t(0), ctypes.c_int64(0)
        L.check(lib.gi_rasterize_size(n, img, cap, ctypes.byref(fwd), ctypes.byref(bwd)), "size")
        state = torch.empty((fwd.value,), dtype=torch.uint8, device="cuda")
        out = torch.full((H, W, 3), -7.0, device="cuda")
        L.check(lib.gi_rasterize_forward(L.ptr(m), L.ptr(l), L.ptr(c), n, img, cap, L.ptr(state), fwd.value,
                                         L.ptr(out), ctypes.byref(pairs), L.stream_handle()), "forward")
        torch.cuda.synchronize()
        assert pairs.value == b.K
        assert torch.equal(out, torch.full_like(out, -7.0) if short else ref)
        assert (gi.device_errors(clear=True) != 0) == short
