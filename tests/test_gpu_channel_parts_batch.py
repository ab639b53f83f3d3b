"""Channel parts where a part has fewer channels than the kernel has classes (65
channels in eight parts: the last has two), alone and in a batch (two parts in the
persistent launch), against the oracle; and the spectrum as the sum over the parts
of the workspace, whenever that is asked for. Tolerance: that of the FP32-accurate
paths, 1e-4."""
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


def workload(sections, per, nx, on_grid, seed=6):
    w = wl.small_mono(seed=seed)
    w.elem_xy, w.elem_section, _ = wl.monostatic_array(0.5, sections, 60.0, per)
    x0, dx = wl.centred_axis(0.2, nx)
    w.grid = dict(w.grid, x0=x0, dx=dx, nx=nx, y0=x0, dy=dx, ny=nx)
    if on_grid:
        w.grid.update(z0=w.z0, dz=w.dz, nz=20)
    return w


def echo_of(w):
    return oracle.synth_echo(w.tx_xy, w.rx_xy, w.z_scan, w.f_hz, w.pts, w.amp).astype(np.complex64)


def error(w, e, img):
    ref = oracle.hybrid_exact(0, w.tx_xy, w.rx_xy, e, w.z_scan, w.f_hz, w.n_pad, w.pix_xy(),
                              w.axis("z"))
    got = img.cpu().numpy().reshape(w.grid["nz"], -1)
    return float(np.linalg.norm(got - ref) / np.linalg.norm(ref))


@pytest.mark.parametrize("sections,per,nx,on_grid,parts", [(5, 13, 24, True, 8), (5, 13, 32, False, 8),
                                                           (3, 19, 16, True, 7)])
def test_parts_of_few_channels(binding, sections, per, nx, on_grid, parts):
    w = workload(sections, per, nx, on_grid)
    e = echo_of(w)
    plan = binding.Plan.from_workload(w, block_config=4)
    img = plan.execute(torch.from_numpy(e).cuda())
    assert plan.workspace(binding.PL_STAGE_BACKPROJECT).shape[0] == parts
    err = error(w, e, img)
    print("%d channels in %d parts: rel L2 %.2e" % (w.n_chan, parts, err))
    assert err < 1e-4


@pytest.mark.parametrize("scenes,tc_launch,extra", [(1, 2, 1), (12, 2, 1), (1, 1, 0), (12, 1, 0)])
def test_batch_of_small_scenes(binding, scenes, tc_launch, extra):
    # `extra`: a launch a scene for the sum of more than two parts
    ws = [workload(5, 13, 32, k % 2 == 0, seed=k) for k in range(scenes)]
    es = [echo_of(w) for w in ws]
    batch = binding.Batch(ws, tc_launch=tc_launch)
    base = 5 * scenes if tc_launch == 2 else 4 * scenes + 1
    assert batch.info["launches_per_execute"] == base + extra * scenes
    imgs = batch.execute([torch.from_numpy(e).cuda() for e in es])
    for w, e, img in zip(ws, es, imgs):
        assert error(w, e, img) < 1e-4


def test_the_parts_sum_to_the_spectrum(binding):
    w = workload(5, 13, 24, False)
    e = torch.from_numpy(echo_of(w)).cuda()
    plan = binding.Plan.from_workload(w, block_config=4)
    plan.execute(e)
    plan.execute(2 * e)
    plan.execute_exact(e)              # a whole spectrum into part 0
    G = plan.workspace(binding.PL_STAGE_BACKPROJECT)
    torch.cuda.synchronize()
    exact = G.sum(0)
    plan.execute(e)
    torch.cuda.synchronize()
    scan = G.sum(0)
    assert G.shape[0] == 8 and not bool(G[1:].any())
    again = plan.workspace(binding.PL_STAGE_BACKPROJECT).sum(0)
    assert torch.equal(again, scan)
    assert float((scan - exact).norm() / exact.norm()) < 1e-4


def test_the_persistent_layout_keeps_two_parts(binding):
    plan = binding.Plan.from_workload(workload(5, 13, 24, False), block_config=4, one_block_per_sm=1)
    assert plan.workspace(binding.PL_STAGE_BACKPROJECT).shape[0] == 2
