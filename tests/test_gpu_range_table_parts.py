"""The range table of 129 to 256 frequencies keeps FP32 operands: the spectrum
operand (the sum of its BF16 parts) against a 64-bit transform, the table against
the 64-bit product of its operands, and the plans that keep the NUFFT (few
channels).

Tolerances. Spectrum: an FP32 FFT of 128 to 360 points, at most 5 stages of some
six roundings of 2^-25 rms each: 1.7e-7 rms; 4e-7 (two BF16 parts of 8 bits round to
2.45e-6 rms). Table: stored as two BF16 parts, 2.45e-6 rms; 3e-6 leaves 1.7e-6 for
the sums of up to 256 complex products (eight truncations of 2^-23 of an atom's
leading sum, 3.5e-7 on average, and FP32 additions)."""
import ctypes

import numpy as np
import pytest

from paper_2109_02842_gb300 import workloads as wl
from test_gpu_range_table import table_values

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    from paper_2109_02842_gb300 import build, binding as b
    build.build()
    b.load()
    return b


def workload(per, n_f, n, n_pad, nx=24, ext=0.14):
    w = wl.small_mono(seed=2)
    w.elem_xy, w.elem_section, _ = wl.monostatic_array(0.5, 1, 40.0, per)
    w.f_hz = wl.uniform_freqs(28e9, 33e9, n_f)
    w.n_scan, w.n_pad = n, n_pad
    w.z0 = -(n - 1) / 2 * w.dz
    x0, dx = wl.centred_axis(ext, nx)
    w.grid = dict(x0=x0, dx=dx, nx=nx, y0=x0, dy=dx, ny=nx, z0=0.0, dz=0.01, nz=2)
    return w


def operand(plan, binding, stage, rows, kp):
    """complex128 [n_pad][rows][kp]: the parts summed."""
    ptr, nbytes = ctypes.c_void_p(), ctypes.c_size_t()
    binding._check(binding.load().pl_plan_workspace(plan._h, stage, ctypes.byref(ptr),
                                                    ctypes.byref(nbytes)))
    n_pad = plan.info["n_pad"]
    planes = nbytes.value // (2 * n_pad * rows * kp)
    raw = torch.as_tensor(binding._DevArray(ptr.value, (n_pad, planes, rows, kp), "<i2"),
                          device="cuda").view(torch.bfloat16).double()
    half = planes // 2
    return torch.complex(raw[:, :half].sum(1), raw[:, half:].sum(1))


@pytest.mark.parametrize("per,n_f,n,n_pad,nx,ext", [
    (128, 129, 64, 128, 24, 0.14), (200, 201, 100, 135, 24, 0.14), (130, 256, 128, 128, 70, 0.45),
    (64, 192, 270, 360, 24, 0.14), (140, 160, 127, 127, 24, 0.14), (65, 193, 100, 256, 148, 0.95)])
def test_operands_and_table(binding, per, n_f, n, n_pad, nx, ext):
    plan = binding.Plan.from_workload(workload(per, n_f, n, n_pad, nx, ext), block_config=4)
    i = plan.info
    assert i["table_exact"] == 1
    g = torch.Generator(device="cuda").manual_seed(n_f)
    e = torch.randn((per, n, n_f), dtype=torch.complex64, device="cuda", generator=g)
    plan.execute(e)
    torch.cuda.synchronize()
    kp = (n_f + 63) // 64 * 64
    A = operand(plan, binding, 16, per, kp)          # PL_WS_RT_OPERAND_A
    S = torch.fft.fft(e.to(torch.complex128), n=n_pad, dim=1).transpose(0, 1)
    err_a = float((A[..., :n_f] - S).abs().pow(2).sum().sqrt() / S.abs().pow(2).sum().sqrt())
    assert bool((A[..., n_f:] == 0).all())
    E = operand(plan, binding, 17,        # PL_WS_RT_OPERAND_E
                (i["table_len"] + 15) // 16 * 16, kp)[:, :i["table_len"]]
    ref = (A @ E.transpose(1, 2)).permute(1, 2, 0).cpu().numpy()          # [c][row][u]
    got = table_values(plan, binding)
    err_t = float(np.linalg.norm(got - ref) / np.linalg.norm(ref))
    print("%d channels, %d f, L %d: spectrum %.2e, table %.2e" % (per, n_f, i["table_len"], err_a,
                                                                  err_t))
    assert err_a < 4e-7
    assert err_t < 3e-6


@pytest.mark.parametrize("per,n_pad,exact", [(63, 360, 0), (64, 360, 1), (16, 1024, 0), (64, 250, 0)])
def test_few_channels_keep_the_nufft(binding, per, n_pad, exact):
    plan = binding.Plan.from_workload(workload(per, 201, 200, n_pad))
    assert plan.info["table_exact"] == exact


def test_a_wait_that_runs_out(binding):
    # (the range table's first stage waits on a barrier nothing completes, for 2 ms)
    w = workload(64, 160, 200, 256)
    e = torch.randn((64, 200, 160), dtype=torch.complex64, device="cuda")
    plan = binding.Plan.from_workload(w, block_config=4, debug_unsatisfiable=2, wait_timeout_us=2000)
    assert plan.info["table_exact"] == 1
    plan.execute(e)
    torch.cuda.synchronize()
    with pytest.raises(binding.PolylineError) as err:
        plan.execute(e)
    assert err.value.status == 8         # PL_ERR_TIMEOUT
    plan.close()
    good = binding.Plan.from_workload(w, block_config=4, wait_timeout_us=2000)
    assert torch.equal(good.execute(e), good.execute(e))
