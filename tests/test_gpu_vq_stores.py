"""Attribute decode at the edges of its store paths: warps of 32 quads and
their remainders, counts that are no multiple of four (the scalar kernel), the
count from which the codebook rows are replicated, positions aligned to 16
but not 32 bytes, small codebooks and indices outside them. The decode is an
exact sum rounded once, so it is compared bit for bit."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gi():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2403_08551_gb300 as m
    m.load()
    return m


def inputs(n, stages, size, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    m16 = (torch.rand((n, 2), generator=g, device="cuda") * 700).half()
    cb = torch.randn((2, stages, size, 3), generator=g, device="cuda")
    idx = torch.randint(0, size, (2, stages, n), generator=g, device="cuda", dtype=torch.uint8)
    return m16, idx, cb


def expected(m16, idx, cb):
    rows = [sum(cb[a, s].double()[idx[a, s].long()] for s in range(cb.shape[1])).float() for a in range(2)]
    return (m16.float(), *rows)


@pytest.mark.parametrize("n,stages,size", [(4, 2, 256), (124, 2, 256), (128, 1, 8), (132, 2, 8), (1021, 2, 256), (4096, 3, 256),
                                           (1199996, 2, 256), (1200000, 2, 256), (1200132, 2, 17), (1200001, 2, 64)])
def test_decode_is_the_exact_sum(gi, n, stages, size):
    m16, idx, cb = inputs(n, stages, size, n)
    for got, want in zip(gi.vq_decode(m16, idx, cb), expected(m16, idx, cb)):
        assert torch.equal(got, want)


@pytest.mark.parametrize("n", [260, 1200040])
def test_decode_into_16_byte_aligned_outputs(gi, n):
    m16, idx, cb = inputs(n, 2, 256, n)
    out = []
    for k in (2, 3, 3):
        buf = torch.full((n * k + 12,), -7.0, device="cuda")
        out.append(buf[4:4 + n * k].view(n, k))  # 16 bytes past a 512-byte boundary
    gi.vq_decode(m16, idx, cb, out=out)
    for got, want in zip(out, expected(m16, idx, cb)):
        assert torch.equal(got, want)
        base = got._base
        assert torch.all(base[:4] == -7) and torch.all(base[4 + got.numel():] == -7)  # nothing written around


def test_index_outside_the_codebook_is_flagged(gi):
    m16, idx, cb = inputs(512, 2, 16, 1)
    gi.device_errors()
    idx[1, 0, 77] = 200
    gi.vq_decode(m16, idx, cb)
    assert gi.device_errors() & 4
