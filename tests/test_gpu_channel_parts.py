"""The tensor-core back-projection of images of few tiles, whose channels go to
up to eight blocks per tile: counts that do not divide, the fewest channels of
each split, heights on the scan grid (the parts summed before the FFT) and off
it (summed as the inverse DFT loads them), against the oracle, bitwise
reproducible. (Two parts add into one spectrum: `parts` is 1 for them.) Tolerance: that of the FP32-accurate paths, 1e-4."""
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


@pytest.mark.parametrize("sections,per,nx,on_grid,parts", [
    (4, 16, 32, False, 8), (3, 21, 24, True, 7), (1, 17, 16, False, 1), (5, 5, 20, True, 3),
    (8, 32, 40, True, 8), (1, 257, 24, True, 1), (4, 30, 64, False, 4)])
def test_channel_parts(binding, sections, per, nx, on_grid, parts):
    w = wl.small_mono(seed=6)
    w.elem_xy, w.elem_section, _ = wl.monostatic_array(0.5, sections, 60.0, per)
    x0, dx = wl.centred_axis(0.2, nx)
    w.grid = dict(w.grid, x0=x0, dx=dx, nx=nx, y0=x0, dy=dx, ny=nx)
    if on_grid:
        w.grid.update(z0=w.z0, dz=w.dz, nz=20)
    echo = oracle.synth_echo(w.tx_xy, w.rx_xy, w.z_scan, w.f_hz, w.pts, w.amp).astype(np.complex64)
    plan = binding.Plan.from_workload(w, block_config=4)
    e = torch.from_numpy(echo).cuda()
    img = plan.execute(e)
    again = plan.execute(e)
    G = plan.workspace(binding.PL_STAGE_BACKPROJECT)
    assert G.shape[0] == parts
    assert torch.equal(img, again)
    ref = oracle.hybrid_exact(0, w.tx_xy, w.rx_xy, echo, w.z_scan, w.f_hz, w.n_pad, w.pix_xy(),
                              w.axis("z"))
    got = img.cpu().numpy().reshape(w.grid["nz"], -1)
    err = float(np.linalg.norm(got - ref) / np.linalg.norm(ref))
    print("parts %d: rel L2 %.2e" % (G.shape[0], err))
    assert err < 1e-4
