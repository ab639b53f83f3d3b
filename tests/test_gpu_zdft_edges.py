"""The FP32 direct DFT over z at the edges of its 32-row, 64-column tiles and
32-term chunks: the inverse transform of an FP32 plan onto heights off the scan
grid against the same sum of the plan's own spectrum in 64 bits.

Tolerance: a sum of at most 67 complex products, 2 x 67 roundings of 2^-24 of
the running sum each: 8e-6 if all had one sign; random signs 7e-7. 4e-6."""
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


@pytest.mark.parametrize("n_pad,nx,ny,nz", [(32, 8, 8, 32), (33, 9, 7, 33), (64, 13, 5, 31),
                                            (67, 1, 1, 1), (40, 65, 1, 2), (65, 16, 12, 65)])
def test_inverse_dft_tiles(binding, n_pad, nx, ny, nz):
    w = wl.small_mono(seed=5)
    w.n_pad = n_pad
    w.grid = dict(x0=-0.03, dx=0.0061, nx=nx, y0=-0.04, dy=0.0061, ny=ny, z0=-0.0431, dz=0.0017,
                  nz=nz)
    g = torch.Generator(device="cuda").manual_seed(n_pad)
    e = torch.randn((w.n_chan, w.n_scan, w.n_f), dtype=torch.complex64, device="cuda", generator=g)
    plan = binding.Plan.from_workload(w, block_config=1)
    img = plan.execute(e).cpu().numpy().astype(np.complex128)
    G = plan.workspace(binding.PL_STAGE_BACKPROJECT).cpu().numpy().astype(np.complex128).sum(0)
    kz = 2 * np.pi * np.fft.fftfreq(n_pad, w.dz)
    ref = np.exp(1j * (w.axis("z")[:, None] - w.z0) * kz) @ G.reshape(n_pad, -1) / n_pad
    err = float(np.linalg.norm(img.reshape(nz, -1) - ref) / np.linalg.norm(ref))
    print("inverse DFT n_pad %d, %d x %d x %d: %.2e" % (n_pad, nx, ny, nz, err))
    assert err < 4e-6
