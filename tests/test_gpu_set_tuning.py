"""amr_get_tuning reports the launch parameters of the next step, also where the
library's rules give them, and amr_set_tuning fixes every one it is given, the
default values too. The rules' values are those of the table beside RhsCfg and
of ghost_ctas / ghost_chunk."""
import numpy as np
import pytest

from synth import workload

pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures('cuda')]

RULES = [('implosion', dict(base_cells=(512, 512, 1), patch=16, levels=1), 32, 4, 16, 128),
         ('implosion', dict(base_cells=(512, 512, 1), patch=8, levels=1), 32, 6, 4, 128),
         ('riemann2d', dict(base_cells=(256, 256, 1), patch=16, levels=1), 64, 8, 16, 128),
         ('blast3d', dict(base_cells=(64, 64, 64), patch=8, levels=1), 32, 4, 16, 192),
         ('blast3d', dict(base_cells=(32, 32, 32), patch=16, levels=1), 32, 2, 16, 128)]


@pytest.mark.parametrize('name,kw,precision,rhs,ghost,cells', RULES)
def test_reported_values_are_those_in_use(name, kw, precision, rhs, ghost, cells):
    from paper_2508_05020_gb300.amr import AMR
    w = workload(name, **kw)
    a, b = AMR(w, precision=precision), AMR(w, precision=precision)
    p = a.tuning()[0]
    assert (p['rhs_ctas_per_sm'], p['ghost_ctas_per_sm'], p['ghost_cells_per_item']) == (rhs, ghost, cells)
    asked = {'rhs_ctas_per_sm': 2, 'ghost_ctas_per_sm': 16, 'ghost_cells_per_item': 128}   # the defaults, explicitly
    b.set_tuning(asked)
    got = b.tuning()[0]
    assert all(got[k] == v for k, v in asked.items())
    a.advance(2, regrid=1)
    b.advance(2, regrid=1)
    for l in range(w['levels']):
        assert np.array_equal(a.get_level(l)[1], b.get_level(l)[1])
    a.close()
    b.close()


def test_a_set_value_stays_when_the_hierarchy_grows():
    from paper_2508_05020_gb300.amr import AMR
    w = workload('riemann2d', base_cells=(128, 128, 1), patch=16, levels=3)
    src = AMR(w, precision=32)
    per = [src.get_level(l) for l in range(3)]
    src.close()
    full = (sum(([l] * len(c) for l, (c, _) in enumerate(per)), []), np.concatenate([c for c, _ in per]),
            np.concatenate([x.ravel() for _, x in per]))
    base = ([0] * len(per[0][0]), per[0][0], per[0][1].ravel())
    for pin in (False, True):
        g = AMR(w, precision=32)
        g.set_state(*base)
        assert g.tuning()[0]['rhs_ctas_per_sm'] == 2     # 64 leaves
        if pin:
            g.set_tuning(g.tuning()[0])
        g.set_state(*full)                               # more than 304 leaves: the rule says 4
        assert g.tuning()[0]['rhs_ctas_per_sm'] == (2 if pin else 4)
        g.close()
