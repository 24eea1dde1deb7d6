"""The positivity test of a prolonged cell's children where the products of its
bound underflow. One cell has children whose squared momenta round to zero while
2 rho E rounds up to the smallest subnormal; in two dimensions and more their
kinetic energy nevertheless exceeds E, so every child has to take the coarse
value. The patch beside it is of ordinary size and keeps its slopes."""
import numpy as np
import pytest

from synth import workload

pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures('cuda')]


def tiny(precision):
    """(rho, m, E) with m^2 = 0.46 s and 2 rho E = 0.55 s, s the smallest
    subnormal: d m^2 / (2 rho E) = 1.7 in 2D, 2.5 in 3D."""
    if precision == 64:
        return 2.0 ** -66, 0.68 * 2.0 ** -537, 0.55 * 2.0 ** -1009
    return 2.0 ** -50, float(np.float32(0.48 * 2.0 ** -74)), float(np.float32(0.55 * 2.0 ** -100))


@pytest.mark.parametrize('precision', [64, 32])
@pytest.mark.parametrize('dim,patch', [(2, 8), (2, 16), (3, 8)])
def test_children_of_a_tiny_cell(dim, patch, precision):
    from oracle.amr import Oracle
    from paper_2508_05020_gb300.amr import AMR
    base = (2 * patch,) + (patch,) * (dim - 1) + (1,) * (3 - dim)
    w = workload('riemann2d' if dim == 2 else 'blast3d', base_cells=base, patch=patch, levels=2,
                 theta_rho=0.05, theta_p=0.05)
    r = Oracle(dict(w, theta_rho=1e9, theta_p=1e9))      # nothing refined: level 0 only
    r.w['theta_rho'] = r.w['theta_p'] = 0.05
    rho, m, E = tiny(precision)
    rng = np.random.default_rng(3)
    i0 = patch // 2
    for k in r.mesh.canonical():
        A = r.U[k]
        cells = A[r.inner()].shape[1:]
        if k[1][0] == 0:
            idx = np.meshgrid(*[np.arange(n) for n in cells], indexing='ij')[::-1]   # x, y, z
            U = np.stack([np.where(idx[0] < 2, 3.0 * rho, rho)] + [4.0 * m * (idx[d] - i0) for d in range(dim)] +
                         [np.full(cells, E)])            # slope 4 m along each dimension: children at -m and +m
        else:
            d = 1.0 + 0.2 * rng.uniform(size=cells)
            v = [0.3 * rng.uniform(size=cells) for _ in range(dim)]
            U = np.stack([d] + [d * q for q in v] + [2.5 + rng.uniform(size=cells)])
        A[r.inner()] = U.astype(np.float32).astype(np.float64) if precision == 32 else U
    c0, x0 = r.get_level(0)
    r.regrid()
    c1, x1 = r.get_level(1)
    assert len(c1) == 2 ** (dim + 1)                     # both patches refined
    g = AMR(w, precision=precision)
    g.set_state([0] * len(c0), c0, x0.ravel(), 0.0)
    g.regrid()
    cg, xg = g.get_level(1)
    g.close()
    assert np.array_equal(cg, c1)
    fine = np.zeros((dim + 2,) + tuple(2 * s for s in reversed(base[:dim])))
    for c, x in zip(cg, xg):                             # the children of the whole level in one array
        fine[(slice(None),) + tuple(slice(c[d] * patch, (c[d] + 1) * patch) for d in reversed(range(dim)))] = x
    kids = fine[(slice(None),) + (slice(2 * i0, 2 * i0 + 2),) * dim].reshape(dim + 2, -1)
    assert np.array_equal(kids, np.array([rho] + [0.0] * dim + [E])[:, None] + np.zeros_like(kids))
    if precision == 64:
        assert np.array_equal(xg, x1)
    else:                                                # the ordinary patch: one rounding of each of d + 1 terms
        right = c1[:, 0] >= 2
        assert np.all(np.abs(xg[right] - x1[right]) <= 4 * 2.0 ** -24 * 4.0)
