"""The comparison algorithms at the edges of their kernels' tiles and chunks:
frequencies staged in several chunks, positions staged in groups with a
remainder, ragged pixel tiles, a remainder of bins, and pixels so far apart
that the exact sum takes its whole-phase kernel.

Tolerance: FP32 sums of N products are off by about sqrt(2 N / 3) 2^-25
relative to the focused image, 1e-6 for the sizes here; a phase is off by at
most 1e-5 rad (kappa delta below 128 rad, rounded three times to 2^-24), with
independent signs; __sincosf by 5e-7. 2e-5 holds all of them."""
import numpy as np
import pytest

import oracle
from paper_2109_02842_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 2e-5


@pytest.fixture(scope="module")
def binding():
    from paper_2109_02842_gb300 import build, binding as b
    build.build()
    b.load()
    return b


def workload(mode=0, n_f=16, n_scan=8, n_pad=8, nx=9, ny=7, nz=3, dx=0.0062, f1=33e9):
    w = wl.small_mono(seed=3)
    if mode == 1:
        xy, sec, ptx, prx, _ = wl.multistatic_array(0.5, 2, 60.0, 1, 7)
        w.mode, w.elem_xy, w.elem_section, w.pair_tx, w.pair_rx = 1, xy, sec, ptx, prx
    else:
        xy, sec, _ = wl.monostatic_array(0.5, 3, 60.0, 7)
        w.elem_xy, w.elem_section = xy, sec
    w.f_hz = np.linspace(28e9, f1, n_f)
    w.n_scan, w.n_pad = n_scan, n_pad
    w.z0 = -(n_scan - 1) / 2 * w.dz
    w.grid = dict(x0=-dx * (nx - 1) / 2, dx=dx, nx=nx, y0=-dx * (ny - 1) / 2, dy=dx, ny=ny,
                  z0=-0.008, dz=0.0081, nz=nz)
    w.pts[:, 2] *= 0.1
    return w


def echo_of(w):
    return oracle.synth_echo(w.tx_xy, w.rx_xy, w.z_scan, w.f_hz, w.pts, w.amp).astype(np.complex64)


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("kw", [
    dict(n_f=2, n_scan=33, n_pad=33), dict(n_f=16, n_scan=1, n_pad=1), dict(n_f=512),
    dict(n_f=530, mode=1), dict(nx=43, ny=3, nz=1), dict(nx=127, ny=1, mode=1),
    dict(n_f=33, n_scan=19, n_pad=20)],
    ids=lambda kw: "-".join("%s%d" % kv for kv in kw.items()))
def test_direct_bp_edges(binding, kw):
    w = workload(**kw)
    e = echo_of(w)
    img = binding.Plan.from_workload(w).execute_bp_direct(torch.from_numpy(e).cuda()).cpu().numpy()
    zz, yy, xx = np.meshgrid(w.axis("z"), w.axis("y"), w.axis("x"), indexing="ij")
    ref = oracle.bp_direct(w.tx_xy, w.rx_xy, e, w.z_scan, w.f_hz,
                           np.stack([xx.ravel(), yy.ravel(), zz.ravel()], 1))
    err = rel(img.ravel(), ref)
    print("direct BP %s: rel L2 %.3e" % (kw, err))
    assert err < TOL


@pytest.mark.parametrize("kw", [
    dict(n_scan=5, n_pad=7), dict(n_f=256), dict(n_f=257, mode=1), dict(n_f=1),
    dict(nx=17, ny=9), dict(nx=33, ny=1, mode=1), dict(dx=0.0102),
    dict(dx=0.05, f1=28.02e9), dict(dx=0.05, mode=1, n_f=257, f1=28.02e9),
    dict(n_scan=1, n_pad=1)],
    ids=lambda kw: "-".join("%s%s" % kv for kv in kw.items()))
def test_exact_sum_edges(binding, kw):
    w = workload(**kw)
    e = echo_of(w)
    # (steps of 5 cm are refused for a wide band: the range table's windows)
    plan = binding.Plan.from_workload(w)
    img = plan.execute_exact(torch.from_numpy(e).cuda()).cpu().numpy()
    ref = oracle.hybrid_exact(w.mode, w.tx_xy, w.rx_xy, e, w.z_scan, w.f_hz, w.n_pad, w.pix_xy(),
                              w.axis("z"))
    err = rel(img.reshape(w.grid["nz"], -1), ref)
    print("exact sum %s: rel L2 %.3e" % (kw, err))
    assert err < TOL
