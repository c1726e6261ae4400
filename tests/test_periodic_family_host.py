"""Which plans take the periodic kernel: pixel/step need not be the compiled
ratio to the last bit, only step through the planes like it (a pixel size or a
step that is rounded to a few digits)."""
import pytest

opm = pytest.importorskip("paper_2211_00645_gb300")


@pytest.mark.parametrize("q", [3, 2])
@pytest.mark.parametrize("off", [0.0, 3e-14, 1e-11, 1e-7])
@pytest.mark.parametrize("shape", [(50, 87, 30.0), (30, 20, 45.0), (200, 512, 35.0)])
def test_plans_near_the_ratio_are_periodic(q, off, shape):
    plan = opm.Plan(shape[0], shape[1], 128, shape[2], 0.1 * q * (1.0 - off), 0.1)
    assert opm.opm_plan_path(plan) == (opm.OPM_PATH_PERIODIC, 1, q)
