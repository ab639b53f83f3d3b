"""The tcgen05 convolution at the shapes the dispatch gives it: wide layers of many
tiles, and layers whose weights leave the column kernel no room, in each width
of the product (16, 32, 64 and 128 output columns), against a 64-bit reference
and, bit for bit, against the general kernel (which takes the same call with
unaligned weights, and sums in the same order).

Tolerance: as for the other kernels, 27 Cin / 16 truncating steps of 2^-23 of
the running sum, random signs: 1e-5 up to Cin = 256."""
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


@pytest.mark.parametrize("dims,cin,cout", [
    ((8, 64, 128), 64, 32), ((4, 32, 128), 64, 128), ((4, 64, 128), 128, 64), ((2, 64, 128), 128, 128),
    ((16, 64, 64), 64, 64), ((1, 3, 128), 128, 32), ((2, 4, 64), 256, 16), ((2, 4, 64), 256, 5),
    ((3, 16, 16), 256, 32), ((2, 16, 128), 128, 64)])
def test_wide_layers(L, dims, cin, cout):
    g = torch.Generator(device="cuda").manual_seed(cin + cout)
    v = dims[0] * dims[1] * dims[2]
    kp = L.lib().pl_nn_padded_k(cin)
    x = torch.randn((v, cin), device="cuda", generator=g).bfloat16()
    w = (torch.randn((cout, kp), device="cuda", generator=g) / (27 * cin) ** 0.5).bfloat16()
    b = torch.randn(cout, device="cuda", generator=g)
    xp = torch.nn.functional.pad(x.double().view(*dims, cin), (0, 0, 1, 1, 1, 1, 1, 1))
    ref = b.double().expand(v, -1).clone()
    for t in range(27):
        part = xp[t // 9:t // 9 + dims[0], t // 3 % 3:t // 3 % 3 + dims[1], t % 3:t % 3 + dims[2]]
        ref += part.reshape(-1, cin) @ w[:, t * cin:(t + 1) * cin].double().T
    y = L.conv3d(x, w, b, dims, cin, cout, False, False)
    err = float((y.double() - ref).norm() / ref.norm())
    print(dims, cin, cout, "%.2e" % err)
    assert err < TOL
    odd = torch.empty(w.numel() + 1, dtype=torch.bfloat16, device="cuda")[1:].view(cout, kp)
    odd.copy_(w)
    for relu, bf16 in ((False, False), (True, True)):
        assert torch.equal(L.conv3d(x, w, b, dims, cin, cout, relu, bf16),
                           L.conv3d(x, odd, b, dims, cin, cout, relu, bf16))
