"""The launches of a step that hold two kernels' work, against the same step
with a launch for each (device timing on): the flux correction with the
restriction of the level below the finest, and the CFL reduction with the
first stage's ghost fill. Both forms run the same device functions in an order
that no result depends on, so every cell is the same to the last bit.

Hierarchies with three and four levels, where leaves border on finer patches
on one and on several sides, patches that are as wide as the domain, periodic,
reflecting and time-dependent boundaries, and more patches than the 1D form in
one launch takes.
"""
import numpy as np
import pytest

from synth import workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope='module', autouse=True)
def cuda():
    torch = pytest.importorskip('torch')
    if not torch.cuda.is_available():
        pytest.skip('no CUDA device')
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)
    yield


CASES = [
    ('shu_osher', dict(base_cells=(2048, 1, 1), patch=8, levels=3)),
    ('riemann2d', dict(base_cells=(48, 32, 1), patch=8, levels=3)),
    ('implosion', dict(base_cells=(32, 32, 1), patch=16, levels=4)),
    ('dmr', dict(base_cells=(64, 16, 1), patch=8, levels=3, flux='hllc')),
    ('shear2d', dict(base_cells=(32, 32, 1), patch=32, levels=3)),
    ('blast3d', dict(base_cells=(16, 8, 16), patch=8, levels=3)),
]


@pytest.mark.parametrize('precision', [64, 32])
@pytest.mark.parametrize('name,kw', CASES)
def test_merged_launches_match_separate_ones(name, kw, precision):
    from paper_2508_05020_gb300.amr import AMR
    w = workload(name, **kw)
    a = AMR(w, precision=precision)
    b = AMR(w, precision=precision)
    b.set_timing(True)
    for regrid in (2, False):
        a.advance(4, regrid=regrid)
        b.advance(4, regrid=regrid)
    assert a.step() == b.step()
    for l in range(w['levels']):
        ca, xa = a.get_level(l)
        cb, xb = b.get_level(l)
        assert np.array_equal(ca, cb) and np.array_equal(xa, xb)
    a.close()
    b.close()
