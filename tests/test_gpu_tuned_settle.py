"""With three levels the step corrects fluxes and restricts in one launch; the
autotuner times that launch for the grid it takes. It holds the flux correction,
so its time is not below the flux correction's alone (by more than the few per
cent of a best of three); the restriction alone takes 0.7 of that here."""
import pytest

from synth import workload

pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures('cuda')]


def test_tuner_times_the_launch_of_the_step():
    from paper_2508_05020_gb300.amr import AMR
    g = AMR(workload('shear2d', base_cells=(256, 256, 1), patch=8, levels=3), precision=64, autotune=True)
    ms = g.tuning()[1]
    g.close()
    assert ms['restrict_ctas_per_sm'] >= 0.93 * ms['reflux_ctas_per_sm'], ms
