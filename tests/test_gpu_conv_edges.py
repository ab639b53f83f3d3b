"""The 3 x 3 x 3 convolution at the edges of its kernels' tiles: rows that
cross the epilogue's warps, rows of more than 128 voxels, padded rows,
remainders of rows and slices, blocks whose share crosses from one column of
the volume into the next, splits of the output channels, and the shapes that
go to the other kernels.

Tolerance: inputs are BF16 and products exact in FP32; a sum of 27 Cin products
runs through at most 27 Cin / 16 truncating tensor-core steps, each at most
2^-23 of the running sum: 1e-5 holds 84 steps of one sign, and the sums here
(random signs) of any length up to Cin = 128."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def L():
    from paper_2109_02842_gb300 import build, learned
    build.build()
    learned.lib()
    return learned


def reference(x, w, b, dims, cin):
    xp = torch.nn.functional.pad(x.double().view(*dims, cin), (0, 0, 1, 1, 1, 1, 1, 1))
    out = b.double().expand(x.shape[0], -1).clone()
    for t in range(27):
        part = xp[t // 9:t // 9 + dims[0], t // 3 % 3:t // 3 % 3 + dims[1], t % 3:t % 3 + dims[2]]
        out += part.reshape(-1, cin) @ w[:, t * cin:(t + 1) * cin].double().T
    return out


@pytest.mark.parametrize("dims,cin,cout", [
    ((1, 1, 1), 16, 16), ((3, 2, 4), 16, 16), ((2, 5, 8), 32, 1), ((4, 7, 13), 16, 32),
    ((3, 11, 40), 16, 2), ((5, 9, 65), 16, 16), ((2, 3, 72), 32, 16), ((6, 10, 128), 16, 16),
    ((3, 2, 129), 16, 15), ((2, 6, 160), 32, 32), ((2, 3, 260), 16, 48), ((40, 33, 24), 16, 16),
    ((7, 40, 16), 64, 32), ((5, 9, 32), 64, 64), ((3, 7, 33), 32, 64), ((4, 18, 16), 64, 128),
    ((3, 5, 20), 48, 80), ((2, 16, 16), 128, 64), ((2, 5, 9), 128, 32), ((2, 3, 5), 96, 20),
    ((160, 2, 6), 16, 16), ((3, 70, 3), 32, 32),
    ((1, 1, 1), 3, 16), ((9, 10, 13), 1, 2), ((3, 33, 81), 3, 16), ((17, 5, 128), 2, 16),
    ((2, 300, 1), 4, 33), ((5, 3, 170), 3, 9), ((4, 7, 6), 5, 16)])
def test_conv_edges(L, dims, cin, cout):
    g = torch.Generator(device="cuda").manual_seed(dims[2] * 1000 + cin)
    v = dims[0] * dims[1] * dims[2]
    kp = L.lib().pl_nn_padded_k(cin)
    x = torch.randn((v, cin), device="cuda", generator=g).bfloat16()
    w = torch.zeros((cout, kp), dtype=torch.bfloat16, device="cuda")
    w[:, :27 * cin] = torch.randn((cout, 27 * cin), device="cuda", generator=g) / (27 * cin) ** 0.5
    b = torch.randn(cout, device="cuda", generator=g)
    ref = reference(x, w[:, :27 * cin], b, dims, cin)
    y = L.conv3d(x, w, b, dims, cin, cout, False, False)
    e = float((y.double() - ref).norm() / ref.norm())
    r = L.conv3d(x, w, b, dims, cin, cout, True, True)
    er = float((r.double() - ref.clamp_min(0)).norm() / ref.clamp_min(0).norm())
    n = L.conv3d(x, w, None, dims, cin, cout, False, False)
    en = float((n.double() - (ref - b.double())).norm() / ref.norm())
    print(dims, cin, cout, "%.2e %.2e %.2e" % (e, er, en))
    assert e < TOL and en < TOL
    assert er < 2 ** -8               # BF16 results: half an ulp, 2^-9, each
    assert torch.equal(y, L.conv3d(x, w, b, dims, cin, cout, False, False))
