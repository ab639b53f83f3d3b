"""Convolutions whose operands are not 16-byte aligned: views a few elements into a
buffer, for x, w and out in turn and together, give the bits of aligned
operands (all kernels sum in the same order)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_2109_02842_gb300 import build, learned
    build.build()
    learned.lib()
    return learned


def moved(t, shift):
    """The same values `shift` elements past an aligned address."""
    b = torch.zeros(t.numel() + shift + 8, dtype=t.dtype, device="cuda")
    v = b[shift:shift + t.numel()].view(t.shape)
    v.copy_(t)
    assert v.data_ptr() % 16 == (shift * t.element_size()) % 16
    return v


@pytest.mark.parametrize("dims,cin,cout", [((3, 5, 7), 3, 16), ((2, 9, 4), 1, 3), ((4, 3, 6), 16, 16),
                                           ((3, 8, 16), 32, 20), ((2, 5, 5), 5, 8), ((2, 4, 64), 64, 64)])
@pytest.mark.parametrize("shifts", [(1, 0, 0), (0, 1, 0), (0, 2, 0), (0, 0, 1), (3, 5, 2), (8, 8, 1)])
@pytest.mark.parametrize("out_bf16", [0, 1])
def test_unaligned_operands(L, dims, cin, cout, shifts, out_bf16):
    g = torch.Generator(device="cuda").manual_seed(cin)
    v = dims[0] * dims[1] * dims[2]
    kp = L.lib().pl_nn_padded_k(cin)
    x = torch.randn((v, cin), device="cuda", generator=g).bfloat16()
    w = torch.zeros((cout, kp), dtype=torch.bfloat16, device="cuda")
    w[:, :27 * cin] = torch.randn((cout, 27 * cin), device="cuda", generator=g) * 0.1
    b = torch.randn(cout, device="cuda", generator=g)
    want = L.conv3d(x, w, b, dims, cin, cout, False, bool(out_bf16))
    xs, ws = moved(x, shifts[0]), moved(w, shifts[1])
    out = moved(torch.full_like(want, 7.0), shifts[2])
    L.B._check(L.lib().pl_nn_conv3d(L._p(xs), L._p(ws), L._p(b), L._p(out), *dims, cin, cout, 0,
                                    out_bf16, L._s()))
    assert torch.equal(out, want)
