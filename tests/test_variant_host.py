"""Which row kernels a plan's launches run is what the plan says, and can be put back."""
import pytest

from paper_2603_29785_gb300 import qtam


@pytest.mark.parametrize("kw", [{}, dict(window="hann"), dict(compute="f64"), dict(n_out=8192, short_dft="auto", envelope="bf16")])
def test_running_variant(kw):
    p = qtam.Plan(4096.0, 262144, (4, 8, 16, 32, 64), 20.0, 2048.0, 128, device=-1, **kw)
    assert qtam.qtam_plan_running_variant(p.handle) == -1             # whatever is registered for the length
    for v in qtam.qtam_plan_variants(p.handle):
        before = qtam.qtam_plan_running_variant(p.handle)
        qtam.qtam_plan_set_variant(p.handle, v)
        assert qtam.qtam_plan_running_variant(p.handle) == v
        qtam.qtam_plan_set_variant(p.handle, before)
        assert qtam.qtam_plan_running_variant(p.handle) == -1


def test_running_variant_arguments():
    with pytest.raises(qtam.QtamError) as e:
        qtam.qtam_plan_running_variant(None)
    assert e.value.status == 1
