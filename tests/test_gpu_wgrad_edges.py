"""Weight and bias gradients of the 3 x 3 x 3 convolution at the edges of the
kernel's tiles: rows past one tile, remainders of rows, steps and segments,
channel counts off the blocks of 8 and 16, unaligned operands.

Tolerance: inputs are BF16 and every product is exact in FP32. A sum of V
products runs in chains of V / 16 tensor-core steps at most, each truncating
to 2^-23 of the running sum: below 200 steps here, 2.4e-5 of the largest
running sum if all had one sign; rounding errors of either sign give
sqrt(200) 2^-23 = 1.7e-6. 1e-5 lies between them."""
import numpy as np
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


def reference(x, gy, dims, cin):
    xp = torch.nn.functional.pad(x.double().view(*dims, cin), (0, 0, 1, 1, 1, 1, 1, 1))
    g = gy.double()
    out = [g.T @ xp[t // 9:t // 9 + dims[0], t // 3 % 3:t // 3 % 3 + dims[1],
                    t % 3:t % 3 + dims[2]].reshape(-1, cin) for t in range(27)]
    return torch.cat(out, 1), g.sum(0)


@pytest.mark.parametrize("dims,cin,cout,shift", [
    ((1, 1, 1), 16, 16, 0), ((3, 1, 5), 3, 2, 0), ((2, 7, 64), 16, 16, 0), ((5, 3, 65), 16, 32, 0),
    ((9, 5, 130), 8, 16, 0), ((4, 33, 17), 24, 20, 0), ((13, 6, 6), 5, 50, 0),
    ((8, 16, 16), 32, 64, 0), ((6, 9, 11), 40, 128, 0), ((3, 300, 1), 16, 64, 0),
    ((2, 3, 31), 16, 16, 1), ((17, 4, 4), 64, 113, 0), ((4, 8, 8), 3, 16, 3)])
def test_wgrad_edges(L, dims, cin, cout, shift):
    g = torch.Generator(device="cuda").manual_seed(dims[0] * 1000 + cin)
    v = dims[0] * dims[1] * dims[2]
    kp = L.lib().pl_nn_padded_k(cin)

    def bf16(n, c):      # `shift` elements past an aligned address
        t = torch.empty(n * c + shift, dtype=torch.bfloat16, device="cuda")
        t[shift:] = torch.randn(n * c, device="cuda", generator=g)
        return t[shift:].view(n, c)

    x, gy = bf16(v, cin), bf16(v, cout)
    gw = torch.full((cout, kp), 2.0, device="cuda")
    gb = torch.full((cout,), 3.0, device="cuda")
    nbytes = L.lib().pl_nn_wgrad_workspace(*dims, cin, cout)
    work = torch.full((nbytes // 4,), float("nan"), device="cuda")

    def call(bias):
        L.B._check(L.lib().pl_nn_conv3d_wgrad(L._p(x), L._p(gy), L._p(gw), L._p(gb) if bias else None,
                                              L._p(work), nbytes, *dims, cin, cout, L._s()))
    call(True)
    rw, rb = reference(x, gy, dims, cin)
    ew = float((gw[:, :27 * cin].double() - 2 - rw).norm() / rw.norm())
    eb = float((gb.double() - 3 - rb).norm() / rb.norm())
    print(dims, cin, cout, "gw %.2e gb %.2e" % (ew, eb))
    assert ew < TOL and eb < TOL
    assert bool((gw[:, 27 * cin:] == 2).all())
    once = gw.clone()
    gw.fill_(2.0)
    call(False)                       # without a bias: the same sums
    assert torch.equal(gw, once) and float((gb.double() - 3 - rb).norm() / rb.norm()) < TOL
