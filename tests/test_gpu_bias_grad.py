"""The bias gradient of gradients of one sign: its rounding errors have no
preferred sign, so that their mean over the channels all but vanishes.

Tolerance: a channel's sum is off by rounding-to-nearest in its last, largest
additions: nine warps, a sixteenth of the parts, then sixteen sums, at most about
30 additions of up to 0.72 2^-23 0.29 (rms, relative) with partial sums that grow
linearly, sqrt(30 / 3) 2.5e-8 = 8e-8; the mean over n >= 64 independent channels
8e-8 / sqrt(n) <= 1e-8, four times that 4e-8. Additions that truncate are off by
2^-25 to 2^-24 of the running sum each, all to one side: 1e-7."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_2109_02842_gb300 import build, learned
    build.build()
    learned.lib()
    return learned


@pytest.mark.parametrize("dims,cin,cout", [((24, 32, 32), 64, 64), ((48, 64, 64), 16, 128),
                                           ((33, 41, 70), 3, 64)])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_one_signed_bias_gradient(L, dims, cin, cout, sign):
    g = torch.Generator(device="cuda").manual_seed(cout)
    v = dims[0] * dims[1] * dims[2]
    x = torch.randn((v, cin), device="cuda", generator=g).bfloat16()
    gy = (sign * torch.rand((v, cout), device="cuda", generator=g)).bfloat16()
    gw = torch.zeros((cout, L.lib().pl_nn_padded_k(cin)), device="cuda")
    gb = torch.zeros(cout, device="cuda")
    nbytes = L.lib().pl_nn_wgrad_workspace(*dims, cin, cout)
    work = torch.empty(nbytes // 4, device="cuda")
    L.B._check(L.lib().pl_nn_conv3d_wgrad(L._p(x), L._p(gy), L._p(gw), L._p(gb), L._p(work), nbytes,
                                          *dims, cin, cout, L._s()))
    ref = gy.double().sum(0)
    rel = (gb.double() - ref) / ref
    mean, worst = float(rel.mean()), float(rel.abs().max())
    print(dims, cin, cout, "mean %.2e worst %.2e" % (mean, worst))
    assert abs(mean) < 4e-8
    assert worst < 4e-7                 # (five times 8e-8)
