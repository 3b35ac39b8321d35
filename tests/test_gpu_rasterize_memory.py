"""What a rasterize node holds between forward and backward, and that nothing
the backward reads lies in the forward's scratch, which later calls reuse."""
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


@pytest.mark.parametrize("W,H,n,T", [(768, 512, 80000, 16), (1100, 700, 80001, 16), (700, 420, 60000, 8)])
def test_held_between_forward_and_backward(gi, W, H, n, T):
    leaf = [torch.from_numpy(a).cuda().requires_grad_() for a in synth.init_gaussians(n, W, H, n + T)]
    up = torch.randn(H, W, 3, device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    torch.autograd.grad(gi.rasterize(*leaf, W, H, T), leaf, up)  # first-call allocations
    rec, rect, cnt = gi.project(*(t.detach() for t in leaf), W, H, T)
    cap = max(8 * n, int(cnt.sum()))
    del rec, rect, cnt
    torch.cuda.synchronize()
    before = torch.cuda.memory_allocated()
    out = gi.rasterize(*leaf, W, H, T)
    held = torch.cuda.memory_allocated() - before
    # the record, key and emission index of each pair of capacity; the count and
    # first pair of each Gaussian; the image; up to 1 MiB each that the allocator
    # does not split off the state's and the image's blocks
    assert held <= 40 * cap + 12 * (n + 1) + 12 * W * H + (2 << 20)
    assert 4 * cap > (2 << 20)  # so that one more array of the capacity shows
    want = torch.autograd.grad(out, leaf, up, retain_graph=True)
    for _ in range(3):  # takes the scratch's memory again
        gi.rasterize(*(2.0 * t for t in leaf), W, H, T)
    got = torch.autograd.grad(out, leaf, up, retain_graph=True)
    for x, y in zip(got, want):
        assert torch.equal(x, y)


def test_one_buffer_form_equals_the_split_one(gi):
    import ctypes
    from paper_2403_08551_gb300 import _lib as L
    lib = L.load()
    W, H, n, T, cap = 200, 150, 1001, 16, 16384
    m, l, c = (torch.from_numpy(a).cuda() for a in synth.init_gaussians(n, W, H, 4))
    img = L.GIImage(W, H, T)
    fwd, bwd, pairs = ctypes.c_size_t(0), ctypes.c_size_t(0), ctypes.c_int64(0)
    L.check(lib.gi_rasterize_size(n, img, cap, ctypes.byref(fwd), ctypes.byref(bwd)), "size")
    state = torch.empty((fwd.value,), dtype=torch.uint8, device="cuda")
    ws = torch.empty((bwd.value,), dtype=torch.uint8, device="cuda")
    out = torch.empty((H, W, 3), device="cuda")
    s = L.stream_handle()
    assert lib.gi_rasterize_forward(L.ptr(m), L.ptr(l), L.ptr(c), n, img, cap, L.ptr(state), fwd.value - 1, L.ptr(out),
                                    ctypes.byref(pairs), s) == 1
    L.check(lib.gi_rasterize_forward(L.ptr(m), L.ptr(l), L.ptr(c), n, img, cap, L.ptr(state), fwd.value, L.ptr(out),
                                     ctypes.byref(pairs), s), "forward")
    up = torch.randn(H, W, 3, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    g = [torch.empty((n, k), device="cuda") for k in (2, 3, 3)]
    L.check(lib.gi_rasterize_backward(L.ptr(state), fwd.value, L.ptr(l), n, img, cap, L.ptr(up), L.ptr(ws), bwd.value,
                                      *(L.ptr(x) for x in g), s), "backward")
    leaf = [t.clone().requires_grad_() for t in (m, l, c)]
    ref = gi.rasterize(*leaf, W, H, T)
    assert torch.equal(out, ref.detach())
    for x, y in zip(g, torch.autograd.grad(ref, leaf, up)):
        assert torch.equal(x, y)
