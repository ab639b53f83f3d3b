"""The learned path's element-wise passes and mean pool: remainders past the
groups of eight, unaligned operands, channel counts off 8. The results are
those of the same roundings in torch, bit for bit (one operation each; the
pool's sum of eight in order, then a rounding)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_2109_02842_gb300 import build, learned
    build.build()
    learned.lib()
    return learned


@pytest.mark.parametrize("n", [1, 7, 8, 9, 2047, 2048 * 8 + 5])
@pytest.mark.parametrize("shift", [0, 1, 2])
def test_elementwise(L, n, shift):
    g = torch.Generator(device="cuda").manual_seed(n)

    def make(dtype):
        t = torch.zeros(n + shift, dtype=dtype, device="cuda")
        t[shift:] = torch.randn(n, device="cuda", generator=g)
        return t[shift:]

    f, y, z, out = make(torch.float32), make(torch.bfloat16), make(torch.bfloat16), make(torch.bfloat16)
    if n > 8:
        f[3], f[5], y[6] = float("nan"), float("inf"), float("nan")
    for op, args, want in ((0, (f, y), torch.where(y.float() > 0, f, torch.zeros_like(f)).bfloat16()),
                           (1, (f, None), f.bfloat16()), (2, (z, y), (z.float() + y.float()).bfloat16())):
        L.elementwise(op, args[0], args[1], out)
        assert torch.equal(torch.nan_to_num(out.float(), nan=7e7), torch.nan_to_num(want.float(), nan=7e7)), op


@pytest.mark.parametrize("dims,c", [((2, 2, 2), 8), ((4, 6, 10), 16), ((2, 4, 2), 3), ((6, 2, 4), 24)])
def test_pool(L, dims, c):
    g = torch.Generator(device="cuda").manual_seed(c)
    x = torch.randn((dims[0] * dims[1] * dims[2], c), device="cuda", generator=g).bfloat16()
    v = x.float().view(dims[0] // 2, 2, dims[1] // 2, 2, dims[2] // 2, 2, c)
    s = torch.zeros_like(v[:, 0, :, 0, :, 0])
    for d in range(8):
        s = s + v[:, d >> 2, :, (d >> 1) & 1, :, d & 1]
    assert torch.equal(L.pool(x, dims, c), (0.125 * s).bfloat16().reshape(-1, c))
