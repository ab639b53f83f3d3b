"""Accuracy of one term of the exact sum, and its time on a slice.

With one channel, one frequency and one bin the spectrum is k S e^{j kappa a}
itself. Its error: the fast sine and cosine are off by at most 2^-21.4 and
2^-21.2 on [-pi, pi] (5.6e-7 together), the reduced phase by half an ulp of pi,
1.2e-7, twice, the coefficient and its two products by 2^-24 each (1.8e-7):
1.0e-6. 1.5e-6 holds it; an FP32 phase of 100 rad would be off by up to 1e-5."""
import math

import numpy as np
import pytest

from paper_2109_02842_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    from paper_2109_02842_gb300 import build, binding as b
    build.build()
    b.load()
    return b


def workload(mode, nx, ny, dx, n_f=1, n_scan=1, per=1):
    w = wl.small_mono(seed=3)
    if mode == 1:
        xy, sec, ptx, prx, _ = wl.multistatic_array(0.5, 1, 20.0, 1, per)
        w.mode, w.elem_xy, w.elem_section, w.pair_tx, w.pair_rx = 1, xy, sec, ptx, prx
    else:
        w.elem_xy, w.elem_section, _ = wl.monostatic_array(0.5, 1, 20.0, per)
    w.f_hz = np.linspace(33e9, 34e9, n_f)
    w.n_scan = w.n_pad = n_scan
    w.z0 = -(n_scan - 1) / 2 * w.dz
    w.grid = dict(x0=-dx * (nx - 1) / 2, dx=dx, nx=nx, y0=-dx * (ny - 1) / 2, dy=dx, ny=ny,
                  z0=w.z0, dz=0.01, nz=1)
    return w


@pytest.mark.parametrize("mode,nx,ny,dx", [(0, 64, 64, 0.0102), (1, 40, 33, 0.0092),
                                           (0, 129, 1, 0.005), (0, 1, 257, 0.002)])
def test_phase_of_one_term(binding, mode, nx, ny, dx):
    w = workload(mode, nx, ny, dx)
    plan = binding.Plan.from_workload(w)
    e = torch.full((w.n_chan, 1, 1), 0.75 - 0.5j, dtype=torch.complex64, device="cuda")
    plan.execute_exact(e)
    got = plan.workspace(binding.PL_STAGE_BACKPROJECT)[0].cpu().numpy().astype(np.complex128)
    k = 2 * math.pi * w.f_hz[0] / wl.C0
    pix = w.pix_xy()
    a = sum(np.hypot(*(pix - np.asarray(q)[0]).T) for q in (w.tx_xy, w.rx_xy))   # both ways
    ref = k * (0.75 - 0.5j) * np.exp(1j * k * a)
    err = float(np.max(np.abs(got.ravel() - ref)) / abs(ref[0]))
    print("one term, mode %d, %d x %d: %.2e" % (mode, nx, ny, err))
    assert err < 1.5e-6


def test_a_slice_costs_what_its_pixels_cost(binding):
    def time_of(nx, ny):
        w = workload(0, nx, ny, 0.0001, n_f=32, n_scan=64, per=48)
        plan = binding.Plan.from_workload(w)
        e = torch.randn((w.n_chan, 64, 32), dtype=torch.complex64, device="cuda")
        img = plan.execute_exact(e)
        best = math.inf
        for _ in range(5):
            t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            t0.record()
            plan.execute_exact(e, img)
            t1.record()
            t1.synchronize()
            best = min(best, t0.elapsed_time(t1))
        return best
    square = time_of(80, 80)
    for nx, ny in ((6400, 1), (1, 6400)):
        assert time_of(nx, ny) < 2 * square     # (idle lanes of a 2-D tile: 8 to 16 times)
