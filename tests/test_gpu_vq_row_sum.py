"""Decodes of three and more stages: the FP32 sum with its errors and the FP64
sum it falls back to, where that matters: ties between two floats, cancellation,
values of very different size, zeros of both signs, denormals, overflow,
infinities and NaN. Bit for bit the FP64 sum in stage order rounded once."""
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


def codebooks(kind, stages, size, g):
    cb = torch.randn((2, stages, size, 3), generator=g, device="cuda")
    if kind == "ties":  # multiples of half a unit of 1 .. 2
        cb = 1 + torch.randint(0, 4, cb.shape, generator=g, device="cuda") * 2.0 ** -23
        cb[:, 1:] = torch.randint(-3, 4, cb[:, 1:].shape, generator=g, device="cuda") * 2.0 ** -24
        cb[:, 2] += torch.randint(-1, 2, cb[:, 2].shape, generator=g, device="cuda") * 2.0 ** -50
    elif kind == "cancel":
        cb[:, 1] = -cb[:, 0] * (1 + torch.randint(-2, 3, cb[:, 0].shape, generator=g, device="cuda") * 2.0 ** -23)
    elif kind == "scales":
        cb *= torch.exp2(torch.randint(-40, 41, cb.shape, generator=g, device="cuda").float())
    elif kind == "zeros":
        cb *= torch.randint(-1, 2, cb.shape, generator=g, device="cuda") == 1
    elif kind == "edge":  # around the smallest term that the FP32 sum takes
        cb = torch.where(cb.abs() < 1, torch.full_like(cb, 2.0 ** -21), torch.ones_like(cb)) * (1 + cb * 2.0 ** -12)
        cb *= torch.randint(-1, 2, cb.shape, generator=g, device="cuda")
    elif kind == "denormal":
        cb *= 2.0 ** -135
    elif kind == "huge":
        cb *= 2.0 ** 126
        cb[..., 0, :], cb[..., 1, :], cb[..., 2, :] = float("inf"), float("-inf"), float("nan")
    return cb.contiguous()


@pytest.mark.parametrize("kind", ["plain", "ties", "cancel", "scales", "zeros", "edge", "denormal", "huge"])
@pytest.mark.parametrize("n,stages,size", [(20000, 3, 64), (20001, 3, 64), (8192, 4, 8), (8192, 8, 256)])
def test_three_and_more_stages(gi, kind, n, stages, size):
    g = torch.Generator("cuda").manual_seed(n + stages)
    cb = codebooks(kind, stages, size, g)
    m16 = torch.zeros((n, 2), device="cuda").half()
    idx = torch.randint(0, size, (2, stages, n), generator=g, device="cuda", dtype=torch.uint8)
    got = gi.vq_decode(m16, idx, cb)[1:]
    for a in range(2):
        want = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
        for s in range(stages):
            want = want + cb[a, s].double()[idx[a, s].long()]
        want = want.float()
        bits, ref = got[a].view(torch.int32), want.view(torch.int32)
        assert torch.all((bits == ref) | (got[a].isnan() & want.isnan()))
