"""Plans of different sizes executed by several host threads at once, each plan on
a stream of its own: every call succeeds and the image keeps the bits it has
alone. The plans share their kernels and differ in the shared memory these take
(scan transforms of 40 and 480 points, table windows, heights)."""
import threading

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


def workload(n_pad, nz, n_f):
    w = wl.small_mono(seed=4)
    w.elem_xy, w.elem_section, _ = wl.monostatic_array(0.5, 2, 60.0, 8)
    w.n_scan, w.n_pad = 24, n_pad
    w.z0 = -11.5 * w.dz
    w.f_hz = wl.uniform_freqs(28e9, 33e9, n_f)
    w.grid = dict(w.grid, nx=16, ny=8, nz=nz, z0=-0.021, dz=0.0013)
    return w


@pytest.mark.parametrize("cfg", [4, 1])
def test_plans_of_different_sizes(binding, cfg):
    jobs = []
    for k, (n_pad, nz, n_f) in enumerate([(40, 9, 16), (480, 96, 16), (40, 9, 30), (480, 96, 40)]):
        w = workload(n_pad, nz, n_f)
        plan = binding.Plan.from_workload(w, block_config=cfg)
        g = torch.Generator(device="cuda").manual_seed(k)
        e = torch.randn((w.n_chan, 24, n_f), dtype=torch.complex64, device="cuda", generator=g)
        alone = plan.execute(e)
        torch.cuda.synchronize()
        jobs.append((plan, torch.cuda.Stream(), e, torch.empty_like(alone), alone))
    bad = []
    gate = threading.Barrier(len(jobs))

    def work(plan, stream, e, img, alone):
        gate.wait()
        try:
            for i in range(3000):
                plan.execute(e, img, stream)
                if i % 50 == 49:
                    stream.synchronize()
                if bad:
                    return
        except binding.PolylineError as err:
            bad.append(str(err))
    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not bad
    for plan, _, _, img, alone in jobs:
        assert torch.equal(img, alone), np.shape(alone)
