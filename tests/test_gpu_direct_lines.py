"""Direct back-projection of volumes whose planes have few pixels, worked on as one
line of voxels: lengths off the blocks of 128, the largest such plane and the
next, the fewest planes, mono- and multistatic, against the oracle, and their time per voxel.

Tolerance: that of the other direct sums at their edges, 2e-5 (FP32 sums of N
products, about sqrt(2 N / 3) 2^-25 relative, 1e-6 here; phases 1e-6 rad)."""
import numpy as np
import pytest

import oracle
from paper_2109_02842_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    from paper_2109_02842_gb300 import build, binding as b
    build.build()
    b.load()
    return b


def workload(mode, nx, ny, nz, n_f=16, per=7, n_scan=8):
    w = wl.small_mono(seed=3)
    if mode == 1:
        xy, sec, ptx, prx, _ = wl.multistatic_array(0.5, 2, 60.0, 1, per)
        w.mode, w.elem_xy, w.elem_section, w.pair_tx, w.pair_rx = 1, xy, sec, ptx, prx
    else:
        w.elem_xy, w.elem_section, _ = wl.monostatic_array(0.5, 2, 60.0, per)
    w.f_hz = np.linspace(28e9, 33e9, n_f)
    w.n_scan = w.n_pad = n_scan
    w.z0 = -(n_scan - 1) / 2 * w.dz
    d = 0.0062
    w.grid = dict(x0=-d * (nx - 1) / 2, dx=d, nx=nx, y0=-d * (ny - 1) / 2, dy=d, ny=ny,
                  z0=-0.02, dz=0.04 / nz, nz=nz)
    w.pts[:, 2] *= 0.1
    return w


@pytest.mark.parametrize("mode,nx,ny,nz,n_f", [(0, 1, 1, 153, 16), (0, 1, 1, 1000, 16), (1, 3, 5, 157, 16),
                                               (0, 8, 8, 155, 130), (1, 64, 1, 153, 3), (0, 13, 5, 153, 16),
                                               (0, 8, 8, 152, 16)])
def test_lines(binding, mode, nx, ny, nz, n_f):
    w = workload(mode, nx, ny, nz, n_f)
    e = oracle.synth_echo(w.tx_xy, w.rx_xy, w.z_scan, w.f_hz, w.pts, w.amp).astype(np.complex64)
    img = binding.Plan.from_workload(w).execute_bp_direct(torch.from_numpy(e).cuda()).cpu().numpy()
    zz, yy, xx = np.meshgrid(w.axis("z"), w.axis("y"), w.axis("x"), indexing="ij")
    ref = oracle.bp_direct(w.tx_xy, w.rx_xy, e, w.z_scan, w.f_hz,
                           np.stack([xx.ravel(), yy.ravel(), zz.ravel()], 1))
    err = float(np.linalg.norm(img.ravel() - ref) / np.linalg.norm(ref))
    print("direct BP %d: %d x %d x %d, %d f: rel L2 %.3e" % (mode, nx, ny, nz, n_f, err))
    assert err < 2e-5


def test_a_line_costs_what_its_voxels_cost(binding):
    def time_of(nx, ny, nz):
        w = workload(0, nx, ny, nz, n_f=32, per=16)
        plan = binding.Plan.from_workload(w)
        e = torch.randn((w.n_chan, 8, 32), dtype=torch.complex64, device="cuda")
        img = plan.execute_bp_direct(e)
        best = float("inf")
        for _ in range(5):
            t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            t0.record()
            plan.execute_bp_direct(e, img)
            t1.record()
            t1.synchronize()
            best = min(best, t0.elapsed_time(t1))
        return best
    cube = time_of(64, 64, 64)
    assert time_of(2, 2, 65536) < 2 * cube       # (a block a plane: 32 times)
