"""The plain sensor in FP64, settled by FP32 bounds where they separate: the
same refinement requests as the oracle at thresholds that the bounds settle, at
thresholds equal to a jump that occurs (the FP64 test decides there), at ones
just beside it, and outside the bounds' range."""
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


def state(name, kw):
    """A state of the workload after a few steps on its base level."""
    from oracle.amr import Oracle
    w = workload(name, levels=2, theta_rho=1e9, theta_p=1e9, **kw)
    r = Oracle(w)                                    # nothing refined: level 0 only
    for _ in range(3):
        r.step()
    return w, r


@pytest.mark.parametrize('name,kw', [('riemann2d', dict(base_cells=(64, 48, 1), patch=16)),
                                     ('sod', dict(base_cells=(64, 1, 1), patch=8)),
                                     ('blast3d', dict(base_cells=(24, 16, 16), patch=8)),
                                     ('dmr', dict(base_cells=(64, 16, 1), patch=8))])
def test_requests_match_oracle_at_every_threshold(name, kw):
    from paper_2508_05020_gb300.amr import AMR
    w, r = state(name, kw)
    c, x = r.get_level(0)
    r.fill_ghosts(r.U, r.t)
    # the largest relative jump of rho of every patch, as the sensor forms it
    f = r.leaf_field(0)
    jumps = []
    for ax in range(f.ndim):
        if f.shape[ax] > 2:
            a, b, m = (np.take(f, range(k, f.shape[ax] - 2 + k), axis=ax) for k in (2, 0, 1))
            jumps.append((np.abs(a - b) / (a + 2 * m + b)).ravel())
    jumps = np.sort(np.concatenate(jumps))
    mid = float(jumps[int(0.97 * len(jumps))])
    for th in (1e-6, 1e-3, 0.05, mid, mid * (1 - 1e-12), mid * (1 + 1e-12), mid * (1 - 1e-6), mid * (1 + 1e-6), 5e3):
        r.w['theta_rho'] = r.w['theta_p'] = th
        want = sorted(tuple(k) for k in [(q[0],) + tuple(q[1]) for q in r.requests()[0]])
        g = AMR(dict(w, theta_rho=th, theta_p=th), precision=64)
        g.set_state([0] * len(c), c, x.ravel(), r.t)
        got = sorted(tuple(int(v) for v in k) for k in g.requests()[0])
        assert got == want, th
        g.close()
