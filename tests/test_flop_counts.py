"""Operation counts of the right-hand sides that the kernels step with (CPU): in the
anisotropic media the FP64 kernels' form of the equations takes fewer operations than that
of the FP32 stages, and the steps' other operations are the same."""
import pytest

from paper_2309_08655_gb300 import rt


@pytest.mark.parametrize("dispersion", [0, 1])
@pytest.mark.parametrize("plasma", [0, 1, 2, 3, 4])
def test_counts_are_those_of_each_form(dispersion, plasma):
    a = rt.rt_flops_per_step(dispersion, plasma)
    b = rt.rt_flops_per_step_mixed(dispersion, plasma)
    assert a[1] - 6 * a[0] == b[1] - 6 * b[0] > 0
    if dispersion == 0:                  # anisotropic
        assert a[0] < b[0]
    assert a[2] == 2 * a[0] + 60


def test_counts_of_the_benchmark_medium():
    assert rt.rt_flops_per_step(0, 0)[:2] == [128.0, 1153.0]
    assert rt.rt_flops_per_step_mixed(0, 0) == [196.0, 1561.0]
    with pytest.raises(Exception):
        rt.rt_flops_per_step_mixed(2, 0)
