"""Prolongation slopes at the domain's sides. A coarse cell at a side takes the
boundary rule's value of the ghost next to it; the double-Mach bottom and top
rules depend on the ghost's own x, which on an x side differs from the cell's.
Two refined patches leave coarse-fine ghosts at both x sides and both y sides,
the rules switch between the ghost and the first cell at both x sides, and the
cells vary so that the slopes there are not zero. Against the oracle with the
same dt: FP64 bit for bit, FP32 within the L1(rho) bar of the parity tests."""
import math

import numpy as np
import pytest

from synth import workload

pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures('cuda')]

X0, X1 = 1.0 / 6.0, 1.0 / 6.0 + 1.0 / math.sqrt(3.0)
BOUNDS = [(('dmr_bottom', 'dmr_top'), ('outflow', 'reflect')),
          (('dmr_top', 'dmr_bottom'), ('dmr_bottom', 'dmr_top')),
          (('reflect', 'outflow'), ('dmr_bottom', 'dmr_top')),
          (('outflow', 'dmr_inflow'), ('dmr_inflow', 'reflect'))]


@pytest.mark.parametrize('precision', [64, 32])
@pytest.mark.parametrize('patch', [8, 16])
@pytest.mark.parametrize('bx,by', BOUNDS)
def test_slopes_take_the_ghosts_own_value(bx, by, patch, precision):
    from oracle.amr import Oracle, dmr_states
    from paper_2508_05020_gb300.amr import AMR
    w = workload('dmr', base_cells=(4 * patch, 4 * patch, 1), patch=patch, levels=2, t_end=0.0,
                 lo=(X0, 0.0, 0.0), hi=(X1, 1.0, 1.0), bc=(bx, by, ('outflow', 'outflow')), theta_rho=1e9, theta_p=1e9)
    r = Oracle(w)
    created = r.mesh.refine([(0, (0, 1, 0)), (0, (3, 2, 0)), (0, (1, 0, 0)), (0, (2, 3, 0))])
    assert len(created) == 16
    rng = np.random.default_rng(7)
    rho, u, v, p = dmr_states(w['gamma'])[1]
    for k in r.mesh.canonical():
        if k not in r.U:
            r.U[k] = np.zeros(r.slot_shape())
        f = rng.uniform(0.9, 1.1, size=(4,) + r.U[k][r.inner()].shape[1:])
        d, a, b, q = rho * f[0], u * f[1], v * f[2], p * f[3]
        U = np.stack([d, d * a, d * b, q / (w['gamma'] - 1.0) + 0.5 * d * (a * a + b * b)])
        r.U[k][r.inner()] = U.astype(np.float32).astype(np.float64)
    levels, coords, data = [], [], []
    for l in range(2):
        c, x = r.get_level(l)
        levels += [l] * len(c)
        coords.append(c)
        data.append(x.reshape(len(c), -1))
    g = AMR(w, precision=precision)
    g.set_state(levels, np.concatenate(coords), np.concatenate(data).ravel(), 0.0)
    for _ in range(2):
        g.step(r.step())
    num = den = 0.0
    for l in range(2):
        _, xg = g.get_level(l)
        _, xr = r.get_level(l)
        if precision == 64:
            assert np.array_equal(xg, xr)
        num += np.sum(np.abs(xg[:, 0] - xr[:, 0]))
        den += np.sum(np.abs(xr[:, 0]))
    g.close()
    assert num <= 1e-5 * den
