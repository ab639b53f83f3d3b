"""A non-finite voxel reaches exactly the weight gradients whose taps touch it:
an infinity or NaN at a corner, an edge, a tile's border or inside the volume
makes the sums of its own input channel non-finite for the taps t with voxel
v - off(t) inside the volume, and leaves every other sum as it is without it."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_2109_02842_gb300 import build, learned
    build.build()
    learned.lib()
    return learned


def gradients(L, x, gy, dims, cin, cout):
    gw = torch.zeros((cout, L.lib().pl_nn_padded_k(cin)), device="cuda")
    gb = torch.zeros(cout, device="cuda")
    nbytes = L.lib().pl_nn_wgrad_workspace(*dims, cin, cout)
    work = torch.empty(nbytes // 4, device="cuda")
    L.B._check(L.lib().pl_nn_conv3d_wgrad(L._p(x), L._p(gy), L._p(gw), L._p(gb), L._p(work), nbytes,
                                          *dims, cin, cout, L._s()))
    return gw[:, :27 * cin].view(cout, 27, cin), gb


@pytest.mark.parametrize("dims,cin,cout", [((4, 9, 70), 16, 16), ((3, 37, 20), 8, 32),
                                           ((5, 6, 7), 3, 2), ((2, 5, 129), 24, 64),
                                           ((3, 300, 1), 16, 16), ((1, 1, 6), 16, 128)])
@pytest.mark.parametrize("value", [float("inf"), float("nan")])
def test_one_bad_voxel(L, dims, cin, cout, value):
    D, H, W = dims
    g = torch.Generator(device="cuda").manual_seed(W)
    x = torch.randn((D * H * W, cin), device="cuda", generator=g).bfloat16()
    gy = (torch.rand((D * H * W, cout), device="cuda", generator=g) + 0.5).bfloat16()   # no zeros
    gw0, gb0 = gradients(L, x, gy, dims, cin, cout)
    spots = {(z, y, c) for z in (0, D - 1) for y in (0, H // 2, H - 1)
             for c in (0, 1, W // 2, 63, 64, 65, W - 2, W - 1) if 0 <= c < W}
    for z, y, c in sorted(spots):
        bad = x.clone()
        ci = (z + y + c) % cin
        bad[(z * H + y) * W + c, ci] = value
        gw, gb = gradients(L, bad, gy, dims, cin, cout)
        hit = torch.zeros((27, cin), dtype=torch.bool, device="cuda")
        for t in range(27):
            # gw[t] pairs voxel v with x at v + (dz, dy, dx) - 1: v of this spot
            v = (z + 1 - t // 9, y + 1 - t // 3 % 3, c + 1 - t % 3)
            hit[t, ci] = all(0 <= a < n for a, n in zip(v, dims))
        assert bool(torch.isfinite(gw[:, ~hit]).all()), (z, y, c)
        assert not bool(torch.isfinite(gw[:, hit]).any()), (z, y, c)
        assert torch.equal(gw[:, ~hit], gw0[:, ~hit]) and torch.equal(gb, gb0)
