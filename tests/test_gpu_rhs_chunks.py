"""The fused RHS where its chunks change: patches cut along y and z, patch
sizes whose faces leave a remainder over the threads, every flux, against the
oracle with the same dt.

FP64 is bit for bit the oracle's arithmetic. FP32: L1(rho) within 1e-5, the
bar of the FP32 parity tests.
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
    ('riemann2d', dict(base_cells=(96, 64, 1), patch=32, levels=2)),
    ('riemann2d', dict(base_cells=(40, 24, 1), patch=8, levels=2, flux='hllc')),
    ('riemann2d', dict(base_cells=(48, 32, 1), patch=16, levels=2, flux='hllc')),
    ('implosion', dict(base_cells=(64, 64, 1), patch=32, levels=2, flux='hybrid')),
    ('shear2d', dict(base_cells=(64, 64, 1), patch=32, levels=2)),
    ('shear2d', dict(base_cells=(40, 40, 1), patch=8, levels=3)),
    ('blast3d', dict(base_cells=(24, 16, 16), patch=8, levels=2, flux='hybrid')),
    ('blast3d', dict(base_cells=(16, 16, 16), patch=8, levels=2, flux='central')),
    ('blast3d', dict(base_cells=(32, 16, 32), patch=16, levels=2, flux='hllc')),
    ('blast3d', dict(base_cells=(16, 16, 16), patch=16, levels=1, flux='central')),
]


@pytest.mark.parametrize('precision', [64, 32])
@pytest.mark.parametrize('name,kw', CASES)
def test_chunked_patches_match_oracle(name, kw, precision):
    from oracle.amr import Oracle
    from paper_2508_05020_gb300.amr import AMR
    w = workload(name, **kw)
    r = Oracle(w)
    g = AMR(w, precision=precision)
    # both start from the oracle's hierarchy and state
    levels, coords, data = [], [], []
    for l in range(w['levels']):
        c, x = r.get_level(l)
        levels += [l] * len(c)
        coords.append(c)
        data.append(x.reshape(len(c), -1))
    g.set_state(levels, np.concatenate(coords), np.concatenate(data).ravel())
    for _ in range(2):
        g.step(r.step())
    num = den = 0.0
    for l in range(w['levels']):
        _, xg = g.get_level(l)
        _, xr = r.get_level(l)
        if precision == 64:
            assert np.array_equal(xg, xr)
        num += np.sum(np.abs(xg[:, 0] - xr[:, 0]))
        den += np.sum(np.abs(xr[:, 0]))
    assert num <= 1e-5 * den
    g.close()


def test_setting_the_reported_defaults_changes_nothing():
    from paper_2508_05020_gb300.amr import AMR
    w = workload('riemann2d', base_cells=(64, 64, 1))
    runs = []
    for again in (False, True):
        g = AMR(w, precision=64)
        if again:
            g.set_tuning(g.tuning()[0])
        g.advance(2, regrid=1)
        runs.append([g.get_level(l)[1] for l in range(w['levels'])])
        g.close()
    assert all(np.array_equal(a, b) for a, b in zip(*runs))
