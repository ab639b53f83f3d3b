"""The exact-sum range table over three and four 64-frequency atoms (129 to 256
frequencies), and the sizes and precisions that keep the NUFFT. Tolerances are
those of the other table tests: 1e-4 for the FP32-level tables."""
import pytest

from paper_2109_02842_gb300 import workloads as wl
from test_gpu_range_table import binding, check_table, echo_of, small_multi  # noqa: F401

pytestmark = pytest.mark.gpu


def workload(mode, n_f, n_pad):
    w = wl.small_mono(seed=2)
    if mode == 0:
        w.elem_xy, w.elem_section, _ = wl.monostatic_array(0.5, 8, 60.0, 16)
    else:
        w = small_multi()
    w.n_pad = n_pad
    w.f_hz = wl.uniform_freqs(28e9, 33e9, n_f)
    return w


@pytest.mark.parametrize("mode,n_f,n_pad,precision,exact", [
    (0, 129, 128, 0, 1), (0, 192, 130, 0, 1), (1, 193, 128, 0, 1), (0, 256, 135, 0, 1),
    (0, 129, 127, 0, 0), (0, 257, 128, 0, 0)])
def test_table_over_more_atoms(binding, mode, n_f, n_pad, precision, exact):  # noqa: F811
    w = workload(mode, n_f, n_pad)
    i = check_table(binding, w, echo_of(w, 2), 1e-4, block_config=4, precision=precision)
    assert i["table_exact"] == exact and i["n_f"] == n_f


def test_bf16_precisions_keep_the_nufft(binding):  # noqa: F811
    for precision in (1, 2):
        w = workload(0, 160, 128)
        i = check_table(binding, w, echo_of(w, 2), 1e-2, block_config=4, precision=precision)
        assert i["table_exact"] == 0
