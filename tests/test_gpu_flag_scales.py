"""The plain sensor in FP64 on states of any scale. Density times a and velocity
times b, both powers of two, scale every term of the sensor by a power of two,
so a scaled state asks for the refinement of the unscaled one, which the oracle
gives. The sensor's FP32 bounds underflow at some of these scales (squared
momenta below the FP32 range, subnormal densities); the FP64 test has to decide
there. The velocity varies strongly where rho and p do not, so that a lost
kinetic energy would look like a pressure jump."""
import numpy as np
import pytest

from synth import workload

pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures('cuda')]

CASES = [('sod', dict(base_cells=(96, 1, 1), patch=8)), ('riemann2d', dict(base_cells=(64, 48, 1), patch=16)),
         ('blast3d', dict(base_cells=(24, 16, 16), patch=8))]


def state(w, r):
    """Level 0 with a smooth density, a pressure jump across one plane and fast
    velocities; set in the oracle r and returned as (coords, conserved values)."""
    dim, N = w['dim'], w['patch']
    for k in r.mesh.canonical():
        _, X = r.cells(k, [0, 0, 0], [N] * 3)
        x = X[0]
        rho = 1.0 + 0.01 * np.sin(6.0 * x)
        p = np.where(x < 0.3, 1.5, 1.0)
        u = [4.0 + 4.0 * np.sin(11.0 * X[d] + 2.0 * x + d) for d in range(dim)]
        E = p / (w['gamma'] - 1.0) + 0.5 * rho * sum(v * v for v in u)
        r.U[k][r.inner()] = np.stack([rho] + [rho * v for v in u] + [E])
    return r.get_level(0)


@pytest.mark.parametrize('a,b', [(0, 0), (-86, 0), (-64, -10), (-130, 30), (-60, 16), (100, -40), (-125, 125),
                                 (60, -80)])
@pytest.mark.parametrize('name,kw', CASES)
def test_requests_do_not_depend_on_the_scale(name, kw, a, b):
    from oracle.amr import Oracle
    from paper_2508_05020_gb300.amr import AMR
    w = workload(name, levels=2, **kw)
    r = Oracle(dict(w, theta_rho=1e9, theta_p=1e9))      # nothing refined: level 0 only
    c, x = state(w, r)
    r.w['theta_rho'] = r.w['theta_p'] = 0.05
    want = sorted((q[0],) + tuple(q[1]) for q in r.requests()[0])
    assert 0 < len(want) < len(c)                        # the jump's patches, not the others
    s = np.array([2.0 ** a] + [2.0 ** (a + b)] * w['dim'] + [2.0 ** (a + 2 * b)])
    g = AMR(dict(w, theta_rho=0.05, theta_p=0.05), precision=64)
    g.set_state([0] * len(c), c, (x * s.reshape((1, -1) + (1,) * w['dim'])).ravel(), 0.0)
    got = sorted(tuple(int(v) for v in k) for k in g.requests()[0])
    g.close()
    assert got == want
