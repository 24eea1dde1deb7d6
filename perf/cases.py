"""Performance cases: the calls a user of the solver makes, over the sizes they are made at.

Three kinds of work, each through its public entry point:

* ``run``: a solver context takes a saved hierarchy (`AMR.set_state`, page-locked
  arrays), advances it by some CFL steps (`AMR.advance`), with or without
  regrids, and gives the new hierarchy back (`AMR.get_level`): a restart, the
  production loop between two outputs, and the output. FP32 fields are handed
  on as FP32 tensors on the GPU, FP64 fields as they come.
* ``grad``: loss and gradient of the learned refinement indicator on device
  rows (`amr_mlp_grad_noalloc`), one call of a caller's own training loop.
* ``train``: the indicator's built-in training (`mlp_train`), host rows in,
  weights and loss history out.

Sizes are those of the named workloads (`synth.workloads`), of the benchmark
and of the indicator's training script, and what lies between them.
"""
import ctypes
import functools
import json
import math

import numpy as np
import torch

from paper_2508_05020_gb300 import amr as amr_api
from paper_2508_05020_gb300.amr import AMR
from synth import mlp_init, workload

G = 3
# operations per face and per cell-stage, by dimension: (Rusanov face, central
# face, cell); the solver's counted numbers (HLLC and hybrid: a Rusanov face)
OPS = {1: (505, 39, 32), 2: (650, 51, 55), 3: (795, 63, 84)}


def listed():
    return [
        # shock tube at its own size, the default precision, a regrid after
        # every step: the smallest hierarchies, launch and host latency
        _run('sod_f64_regrid', 'sod', (64,), 3, 16, 64, steps=32, regrid=1),
        # shock-entropy problem at its own size, FP32, fixed mesh: launch
        # latency of the step alone
        _run('shu_osher_f32', 'shu_osher', (256,), 4, 32, 32, steps=32),
        # four-quadrant problem at its own size, the default precision, a
        # regrid after every step: an ordinary 2D run
        _run('riemann2d_f64_regrid', 'riemann2d', (256, 256), 3, 16, 64, steps=4, regrid=1),
        # double Mach reflection at the reduced size of the tests, FP64, the
        # HLLC flux option, four levels, time-dependent boundary
        _run('dmr_f64_hllc', 'dmr', (128, 32), 4, 16, 64, flux='hllc', steps=8, regrid=2),
        # the implosion benchmark, FP32, periodic, fixed mesh between regrids
        _run('implosion_f32', 'implosion', (256, 256), 3, 16, 32, steps=16),
        # the uniform 2560^2 grid of the stage-update timing, one level, FP32
        _run('uniform2560_f32', 'implosion', (2560, 2560), 1, 16, 32, steps=16),
        # shear layers with the shock-free central schemes, FP32
        _run('shear2d_f32_central', 'shear2d', (256, 256), 3, 16, 32, flux='central', steps=16),
        # the 3D blast as the benchmark runs it: 128^3 base, FP32, learned
        # flags, a regrid every 4 steps (the whole call)
        _run('blast3d_f32_learned', 'blast3d', (128, 128, 128), 3, 16, 32, flagger='mlp', steps=16, regrid=4, pool=4096),
        # the same gas on small patches with the hybrid flux, ragged base (6 x 5 x 7 patches), fixed mesh
        _run('blast3d_f32_patch8_hybrid', 'blast3d', (48, 40, 56), 3, 8, 32, flux='hybrid', steps=8),
        # the 3D blast at the tests' reduced size in the default precision
        _run('blast3d_f64_regrid', 'blast3d', (32, 32, 32), 3, 16, 64, steps=2, regrid=1),
        # gradient of the 3D indicator at the largest row count of the call
        {'name': 'grad_d3_2048', 'kind': 'grad', 'dim': 3, 'rows': 2048},
        # training of the 3D indicator, the script's batch size, a ragged number of rows
        {'name': 'train_d3', 'kind': 'train', 'dim': 3, 'rows': 4700, 'batch': 512, 'epochs': 1},
    ]


def _run(name, wl, base, levels, patch, precision, flux='rusanov', flagger='plain', steps=8, regrid=0, pool=0):
    c = {'kind': 'run', 'workload': wl, 'levels': levels, 'patch': patch, 'precision': precision, 'flux': flux,
         'flagger': flagger, 'steps': steps, 'regrid': regrid, 'pool': pool}
    for d, n in enumerate(base):
        c['base%d' % d] = n
    if name:
        c['name'] = name
    return c


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(['run1', 'run2', 'run2', 'run3', 'run3', 'grad', 'train'])
    if kind == 'grad':
        return {'kind': 'grad', 'dim': rng.choice([1, 2, 3]), 'rows': _log(rng, 33, 2048)}
    if kind == 'train':
        return {'kind': 'train', 'dim': rng.choice([1, 2, 3]), 'rows': _log(rng, 1100, 8000),
                'batch': rng.choice([256, 512, 1000]), 'epochs': 1}
    f64 = rng.random() < 0.5
    # FP64 runs regrid as the production loop does; FP32 runs take the steps between two regrids
    kw = dict(steps=rng.randint(2, 12), regrid=rng.choice([1, 2, 4]) if f64 else 0)
    prec = 64 if f64 else 32
    if kind == 'run1':
        wl = rng.choice(['sod', 'shu_osher', 'density_wave'])
        patch = rng.choice([8, 16, 32])
        return _run('', wl, (patch * _log(rng, 3, 64),), rng.randint(1, 4), patch, prec,
                    flux=rng.choice(['rusanov', 'hllc', 'hybrid']), **kw)
    if kind == 'run2':
        wl = rng.choice(['riemann2d', 'dmr', 'implosion', 'shear2d'])
        patch = rng.choice([8, 16, 16, 32])
        n = _log(rng, 64, 200 if f64 else 512) // patch + 1
        base = (patch * (4 * n), patch * n) if wl == 'dmr' else (patch * n, patch * (n + rng.randint(0, 2)))
        if wl == 'dmr':
            base = (patch * max(4, 2 * n), patch * max(1, n // 2))
        flux = 'central' if wl == 'shear2d' else rng.choice(['rusanov', 'rusanov', 'hllc', 'hybrid'])
        return _run('', wl, base, rng.randint(1, 3), patch, prec, flux=flux, **kw)
    patch = rng.choice([8, 16, 16])
    n = max(2, _log(rng, 24, 32 if f64 else 80) // patch)
    base = (patch * n, patch * (n + rng.randint(0, 1)), patch * n)
    kw['steps'] = min(kw['steps'], 2) if f64 else kw['steps']
    return _run('', 'blast3d', base, rng.randint(1, 3) if not f64 else rng.randint(1, 2), patch, prec,
                flux=rng.choice(['rusanov', 'rusanov', 'hllc', 'hybrid']), **kw)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _workload(case, seed):
    base = tuple(case.get('base%d' % d, 1) for d in range(3))
    w = workload(case['workload'], base_cells=base, levels=case['levels'], patch=case['patch'], flux=case['flux'])
    w['seed'] = int(seed)
    w['t_end'] = 0.0                                     # no clipping: every step is a CFL step
    return w


def _pinned(n):
    return torch.empty(max(int(n), 1), dtype=torch.float64, pin_memory=True).numpy()


def _context(case, seed):
    """The solver context and the hierarchy it starts with."""
    w = _workload(case, seed)
    learned = case['flagger'] == 'mlp'
    kw = {}
    if learned:
        kw = dict(mlp_weights=np.load('paper_2508_05020_gb300/weights/indicator_d%d_diag_k4.npy' % w['dim']).astype(np.float32),
                  mlp_keep_margin=12.0)
    sim = AMR(w, precision=case['precision'], flagger=case['flagger'], max_patches=case['pool'], **kw)
    return w, sim


def _saved(case, seed, w, sim):
    """A saved hierarchy: the workload's initial one, its gas scaled by a
    smooth seeded field of half a per cent (velocity and temperature stay)."""
    dim, N = w['dim'], w['patch']
    coords = [sim.get_level(l, data=False)[0] for l in range(w['levels'])]
    counts = [len(c) for c in coords]
    per = sim.nv * N ** dim
    data = _pinned(sum(counts) * per)
    r = np.random.default_rng(seed)
    k = r.integers(1, 4, size=dim)
    phase = r.uniform(0.0, 2.0 * math.pi, size=dim)
    o = 0
    for l, n in enumerate(counts):
        if not n:
            continue
        block = data[o * per:(o + n) * per].reshape((n, sim.nv) + (N,) * dim)
        sim.get_level(l, out=block)
        f = np.ones((n, 1) + (1,) * dim)
        for d in range(dim):
            cells = w['base_cells'][d] << l
            x = (coords[l][:, d:d + 1] * N + np.arange(N)[None, :] + 0.5) / cells
            shape = [n, 1] + [1] * dim
            shape[1 + dim - d] = N
            f = f * (1.0 + 0.005 / dim * np.sin(2.0 * math.pi * k[d] * x + phase[d])).reshape(shape)
        block *= f
        if case['precision'] == 32:
            block[...] = block.astype(np.float32)
        o += n
    levels = np.concatenate([np.full(n, l, dtype=np.int32) for l, n in enumerate(counts)])
    return levels, np.concatenate(coords).astype(np.int32), data


def _rows(case, seed):
    """Rows as the indicator is trained on: centre-normalised 5^d stencils of
    planar fronts of random direction, place, width and strength, and the label
    of a jump at the centre."""
    dim, n = case['dim'], case['rows']
    g = np.random.default_rng(seed)
    nrm = g.normal(size=(n, dim))
    nrm /= np.linalg.norm(nrm, axis=1, keepdims=True)
    off = np.stack(np.meshgrid(*[np.arange(-2, 3)] * dim, indexing='ij'), axis=-1).reshape(-1, dim)[:, ::-1]
    s = nrm @ off.T + g.uniform(-6.0, 6.0, size=(n, 1))
    amp = np.exp(g.normal(-2.5, 1.2, size=(n, 1)))
    front = np.tanh(s / np.exp(g.normal(0.3, 0.5, size=(n, 1))))
    rho, p = 1.0 + 0.4 * amp / (1.0 + amp) * front, 1.0 + 0.6 * amp / (1.0 + amp) * front
    u = 0.5 * amp / (1.0 + amp) * front + g.normal(0.0, 0.5, size=(n, 1))
    c = len(off) // 2
    c0 = np.sqrt(1.4 * p[:, c:c + 1] / rho[:, c:c + 1])
    X = np.empty((n, len(off), dim + 2), dtype=np.float32)
    X[:, :, 0] = rho / rho[:, c:c + 1] - 1.0
    X[:, :, dim + 1] = p / p[:, c:c + 1] - 1.0
    for d in range(dim):
        X[:, :, 1 + d] = u * nrm[:, d:d + 1] / c0
    y = (np.abs(s[:, c]) < 2.0) & (amp[:, 0] > 0.08)
    y[0] = True
    pw = float((n - y.sum()) / max(y.sum(), 1))
    return X.reshape(n, -1), y.astype(np.float32), pw


def _weights(dim, seed):
    p = mlp_init(seed, 5 ** dim * (dim + 2))
    return np.concatenate([p[k].ravel() for k in ('W1', 'b1', 'W2', 'b2', 'W3', 'b3')]).astype(np.float32)


def prepare(case, seed):
    if case['kind'] == 'run':
        w, sim = _context(case, seed)
        levels, coords, data = _saved(case, seed, w, sim)
        # room for the hierarchy to grow by half before the next output
        room = int(data.size * 1.5) + 64 * sim.nv * w['patch'] ** w['dim']
        return {'case': case, 'sim': sim, 'w': w, 'levels': levels, 'coords': coords, 'data': data, 'out': _pinned(room)}
    X, y, pw = _rows(case, seed)
    wts = _weights(case['dim'], seed)
    if case['kind'] == 'train':
        return {'case': case, 'X': X, 'y': y, 'pw': pw, 'w': wts}
    dev = [torch.from_numpy(a).cuda() for a in (X, y, wts)]
    return {'case': case, 'X': dev[0], 'y': dev[1], 'w': dev[2], 'pw': pw, 'lib': amr_api.load(),
            'grad': torch.empty_like(dev[2]), 'loss': torch.empty(1, device='cuda')}


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    case = state['case']
    if case['kind'] == 'grad':
        p = lambda t: ctypes.c_void_p(t.data_ptr())     # noqa: E731
        rc = state['lib'].amr_mlp_grad_noalloc(case['dim'], p(state['X']), p(state['y']), case['rows'],
                                               ctypes.c_float(state['pw']), p(state['w']), p(state['grad']),
                                               p(state['loss']), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if rc != 0:
            raise RuntimeError('amr_mlp_grad_noalloc: %d' % rc)
        return {'grad': state['grad'], 'loss': state['loss']}
    if case['kind'] == 'train':
        w, hist = amr_api.mlp_train(case['dim'], state['X'], state['y'], state['pw'], state['w'], case['epochs'],
                                    case['batch'], 2e-3)
        return {'weights': w, 'loss': hist}
    sim, w, buf = state['sim'], state['w'], state['out']
    sim.set_state(state['levels'], state['coords'], state['data'], 0.0)
    sim.advance(case['steps'], regrid=case['regrid'])
    N, dim, o, out = w['patch'], w['dim'], 0, []
    for l in range(w['levels']):
        coords, _ = sim.get_level(l, data=False)
        shape = (len(coords), sim.nv) + (N,) * dim
        n = math.prod(shape)
        if o + n > buf.size:                             # the hierarchy outgrew the buffer
            grown = _pinned(2 * (o + n))
            grown[:o] = buf[:o]
            state['out'] = buf = grown
        if n:
            sim.get_level(l, out=buf[o:o + n].reshape(shape))
        out.append((coords, o, n, shape))
        o += n
    if case['precision'] == 64:
        return {'coords': [c for c, _, _, _ in out], 'cells': [buf[a:a + n].reshape(s) for _, a, n, s in out]}
    dev = torch.from_numpy(buf[:o]).cuda(non_blocking=True).float()
    return {'coords': [c for c, _, _, _ in out], 'cells': [dev[a:a + n].reshape(s) for _, a, n, s in out]}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _sizes(key):
    """(patches, leaf patches) of the saved hierarchy (the mesh of one seed)."""
    case = json.loads(key)
    w, sim = _context(case, 1)
    have = [{tuple(c) for c in sim.get_level(l, data=False)[0]} for l in range(w['levels'])]
    sim.close()
    total = sum(len(h) for h in have)
    covered = sum(len({tuple(x // 2 for x in c) for c in h}) for h in have[1:])
    return total, total - covered


def work(case):
    if case['kind'] == 'run':
        total, leaves = _sizes(json.dumps({k: v for k, v in case.items() if k != 'name'}, sort_keys=True))
        dim = sum(1 for d in range(3) if 'base%d' % d in case)
        N, nv, size = case['patch'], dim + 2, case['precision'] // 8
        cells = leaves * N ** dim
        rus, cen, cell = OPS[dim]
        face = cen if case['flux'] == 'central' else rus
        flops = 3 * (cells * cell + leaves * dim * N ** (dim - 1) * (N + 1) * face)
        # saved hierarchy in and out (FP64 values); a step reads the state and
        # writes it, stages two and three each read two states and write one
        return {'bytes': 2 * total * nv * N ** dim * 8 + case['steps'] * 8 * nv * size * cells,
                'flops': case['steps'] * flops}
    dim, n = case['dim'], case['rows']
    K = 5 ** dim * (dim + 2)
    nw = 64 * K + 64 + 64 * 64 + 64 + 64 + 1
    # forward, and backward to the weights of both layers and through the second
    flops = 2 * n * (2 * 64 * K + 3 * 64 * 64 + 3 * 64)
    if case['kind'] == 'grad':
        return {'bytes': 4 * (n * (K + 1) + 2 * nw + 1), 'flops': flops}
    b = min(case['batch'], n)
    used = n // b * b * case['epochs']
    # rows in; every step reads its rows, the weights and the two moments, and writes the last three
    return {'bytes': 4 * (n * (K + 1) + used * (K + 1) + used // b * 6 * nw + 2 * nw), 'flops': flops / n * used}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------
def exact(case, seed):
    if case['kind'] == 'grad':
        X, y, pw = _rows(case, seed)
        g, loss = _grad64(case['dim'], *[torch.from_numpy(a).double().cuda() for a in (X, y)], pw,
                          torch.from_numpy(_weights(case['dim'], seed)).double().cuda())
        return {'grad': g, 'loss': loss.reshape(1)}
    if case['kind'] == 'train':
        return _train64(case, seed)
    if case['regrid']:
        return None                                      # the mesh, remade on the way, decides what comes out
    w, sim = _context(case, seed)
    levels, coords, data = _saved(case, seed, w, sim)
    sim.close()
    got = _advance64(w, levels, coords, data, case['steps'])
    return {'coords': [None for _ in got], 'cells': got}


def _grad64(dim, X, y, pw, w):
    K = X.shape[1]
    w = w.detach().clone().requires_grad_(True)
    W1, b1, W2, b2, W3, b3 = torch.split(w, [64 * K, 64, 64 * 64, 64, 64, 1])
    h = torch.relu(X @ W1.reshape(64, K).T + b1)
    h = torch.relu(h @ W2.reshape(64, 64).T + b2)
    z = h @ W3 + b3
    sp = torch.nn.functional.softplus
    loss = (pw * y * sp(-z) + (1.0 - y) * sp(z)).mean()
    loss.backward()
    return w.grad, loss.detach()


def _train64(case, seed):
    X, y, pw = _rows(case, seed)
    X, y = (torch.from_numpy(a).double().cuda() for a in (X, y))
    w = torch.from_numpy(_weights(case['dim'], seed)).double().cuda()
    n, B = len(X), min(case['batch'], len(X))
    m, v = torch.zeros_like(w), torch.zeros_like(w)
    hist, step = [], 0
    mask = (1 << 64) - 1
    for ep in range(case['epochs']):
        # the epoch's order: r -> (a r + b) mod n from a SplitMix64 draw of seed 1
        z = (1 + (ep + 1) * 0x9E3779B97F4A7C15) & mask
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        z ^= z >> 31
        a = z % n | 1
        while math.gcd(a, n) != 1:
            a += 2
        idx = torch.from_numpy((a % n * np.arange(n) + (z >> 32) % n) % n).cuda()
        loss = 0.0
        for bi in range(n // B):
            rows = idx[bi * B:(bi + 1) * B]
            g, one = _grad64(case['dim'], X[rows], y[rows], pw, w)
            loss = loss + one / (n // B)
            step += 1
            m = 0.9 * m + 0.1 * g
            v = 0.999 * v + 0.001 * g * g
            w = w - 2e-3 * (m / (1.0 - 0.9 ** step)) / (torch.sqrt(v / (1.0 - 0.999 ** step)) + 1e-8)
        hist.append(loss)
    return {'weights': w, 'loss': torch.stack(hist)}


def _primitives(U, dim, gamma):
    u = [U[1 + d] / U[0] for d in range(dim)]
    p = (gamma - 1.0) * (U[dim + 1] - 0.5 * U[0] * sum(x * x for x in u))
    return u, p, p / U[0]


def _weno(a, b, c, d, e):
    t = (a - 2 * b + c, b - 2 * c + d, c - 2 * d + e)
    s = (a - 4 * b + 3 * c, b - d, 3 * c - 4 * d + e)
    q = ((3 * a - 10 * b + 15 * c) / 8, (-b + 6 * c + 3 * d) / 8, (3 * c + 6 * d - e) / 8)
    al = [k / (1e-6 + 13.0 / 12.0 * x * x + 0.25 * y * y) ** 2 for k, x, y in zip((0.0625, 0.625, 0.3125), t, s)]
    return (al[0] * q[0] + al[1] * q[1] + al[2] * q[2]) / (al[0] + al[1] + al[2])


def _side(p, un, ut, T, gamma):
    rho, c = p / T, torch.sqrt(gamma * T)
    E = p / (gamma - 1.0) + 0.5 * rho * (un * un + sum(x * x for x in ut))
    m = rho * un
    return [rho, m] + [rho * x for x in ut] + [E], [m, m * un + p] + [m * x for x in ut] + [(E + p) * un], c


def _weno_flux(p, un, ut, T, gamma, hllc):
    """Flux between nodes 2 and 3 of six-node pencils: characteristic WENO5 and Rusanov or HLLC."""
    pb, Tb = 0.5 * (p[2] + p[3]), 0.5 * (T[2] + T[3])
    rb = pb / Tb
    z, kap = rb * torch.sqrt(gamma * Tb), (gamma - 1.0) / (gamma * rb)
    fields = [[p[k] - z * un[k] for k in range(6)], [T[k] - kap * p[k] for k in range(6)],
              [p[k] + z * un[k] for k in range(6)]] + ut
    st = []
    for nodes, near in (((0, 1, 2, 3, 4), 2), ((5, 4, 3, 2, 1), 3)):
        w = [_weno(*[f[k] for k in nodes]) for f in fields]
        ps, us = 0.5 * (w[0] + w[2]), (w[2] - w[0]) / (2 * z)
        st.append((near, ps, us, w[1] + kap * ps, w[3:]))
    bad = ~((st[0][1] > 0) & (st[0][3] > 0) & (st[1][1] > 0) & (st[1][3] > 0))
    sides = []
    for near, ps, us, Ts, uts in st:
        pick = lambda x, y: torch.where(bad, y, x)       # noqa: E731
        sides.append((pick(ps, p[near]), pick(us, un[near]), [pick(x, f[near]) for x, f in zip(uts, ut)], pick(Ts, T[near])))
    (UL, FL, cL), (UR, FR, cR) = (_side(*s, gamma) for s in sides)
    (pL, uL, tL, _), (pR, uR, tR, _) = sides
    if not hllc:
        S = torch.maximum(cL + uL.abs(), cR + uR.abs())
        return [0.5 * (a + b) - 0.5 * S * (d - c) for a, b, c, d in zip(FL, FR, UL, UR)]
    wL, wR = torch.minimum(uL - cL, uR - cR), torch.maximum(uL + cL, uR + cR)
    aL, aR = UL[0] * (wL - uL), UR[0] * (wR - uR)
    sM = (pR - pL + aL * uL - aR * uR) / (aL - aR)
    out = []
    star = []
    for U, a, wv, uu, tt, pp in ((UL, aL, wL, uL, tL, pL), (UR, aR, wR, uR, tR, pR)):
        f = a / (wv - sM)
        star.append([f, f * sM] + [f * x for x in tt] + [f * (U[-1] / U[0] + (sM - uu) * (sM + pp / a))])
    for v in range(len(UL)):
        x = torch.where(sM >= 0, FL[v] + wL * (star[0][v] - UL[v]), FR[v] + wR * (star[1][v] - UR[v]))
        x = torch.where(~(sM >= 0) & ~(wR > 0), FR[v], x)
        out.append(torch.where(wL >= 0, FL[v], x))
    return out


def _central_flux(p, un, ut, T, gamma):
    """Euler flux of the fourth-order mid value of four-node pencils."""
    mid = lambda f: (9 * (f[1] + f[2]) - (f[0] + f[3])) / 16     # noqa: E731
    pm, Tm = mid(p), mid(T)
    bad = ~((pm > 0) & (Tm > 0))
    pick = lambda f, m: torch.where(bad, 0.5 * (f[1] + f[2]), m)   # noqa: E731
    return _side(pick(p, pm), pick(un, mid(un)), [pick(f, mid(f)) for f in ut], pick(T, Tm), gamma)[1]


class _Dense64:
    """A hierarchy as one dense array per level, (variable, z, y, x), with
    masks of the cells that patches hold and of those that finer ones cover."""

    def __init__(self, w, levels, coords):
        self.w, self.dim, self.N, self.L, self.gamma = w, w['dim'], w['patch'], w['levels'], w['gamma']
        self.coords = [coords[levels == l] for l in range(self.L)]
        self.n = [[w['base_cells'][d] << l for d in range(self.dim)] for l in range(self.L)]
        self.dx = [[(w['hi'][d] - w['lo'][d]) / self.n[l][d] for d in range(self.dim)] for l in range(self.L)]
        self.has = [self._cells(self.coords[l], l) for l in range(self.L)]
        self.cov = [self._cells(np.unique(self.coords[l + 1] // 2, axis=0), l) if l + 1 < self.L and len(self.coords[l + 1])
                    else torch.zeros_like(self.has[l]) for l in range(self.L)]

    def _cells(self, coords, l):
        m = torch.zeros([k // self.N for k in self.n[l]][::-1], dtype=torch.bool, device='cuda')
        if len(coords):
            m[tuple(torch.from_numpy(coords[:, d].astype(np.int64)).cuda() for d in reversed(range(self.dim)))] = True
        for ax in range(self.dim):
            m = m.repeat_interleave(self.N, dim=ax)
        return m

    def _blocks(self, U):
        """(patches along each axis.., variable, N..) view of a dense array."""
        for ax in range(1, self.dim + 1):
            U = U.unfold(ax, self.N, self.N)
        return U

    def dense(self, levels, data):
        N, dim, nv = self.N, self.dim, self.dim + 2
        out = []
        data = torch.from_numpy(np.ascontiguousarray(data)).cuda().reshape((-1, nv) + (N,) * dim)
        for l in range(self.L):
            U = torch.zeros([nv] + self.n[l][::-1], dtype=torch.float64, device='cuda')
            if len(self.coords[l]):
                at = tuple(torch.from_numpy(self.coords[l][:, d].astype(np.int64)).cuda() for d in reversed(range(dim)))
                rows = torch.from_numpy(np.nonzero(levels == l)[0]).cuda()
                self._blocks(U)[(slice(None),) + at] = data[rows].transpose(0, 1)
            out.append(U)
        return out

    def patches(self, U):
        out = []
        for l in range(self.L):
            at = tuple(torch.from_numpy(self.coords[l][:, d].astype(np.int64)).cuda() for d in reversed(range(self.dim)))
            out.append(self._blocks(U[l])[(slice(None),) + at].transpose(0, 1).contiguous())
        return out

    def padded(self, U, l, t):
        """Three ghost layers by the boundary rules, one dimension after the other."""
        for d in range(self.dim):
            ax = self.dim - d
            n = U.shape[ax]
            ends = []
            for side in (0, 1):
                kind = self.w['bc'][d][side]
                if kind == 'periodic':
                    g = U.narrow(ax, n - G if side == 0 else 0, G)
                elif kind == 'outflow':
                    g = U.narrow(ax, 0 if side == 0 else n - 1, 1).repeat_interleave(G, dim=ax)
                else:
                    g = U.narrow(ax, 0 if side == 0 else n - G, G).flip(ax).clone()
                    g[1 + d] = -g[1 + d]
                    if kind.startswith('dmr'):
                        pre, post = _dmr_states(self.gamma)
                        x = torch.arange(g.shape[-1], dtype=torch.float64, device='cuda')
                        x = self.w['lo'][0] + (x - G + 0.5) * self.dx[l][0]    # (the inflow takes no account of it)
                        lim = 1e30 if kind == 'dmr_inflow' else 1 / 6 + (0.0 if kind == 'dmr_bottom' else (1 + 20 * t) / math.sqrt(3))
                        behind = (x < lim).expand(g.shape[1:])
                        for v in range(4):
                            fixed = torch.where(behind, post[v], pre[v])
                            g[v] = torch.where(behind, fixed, g[v]) if kind == 'dmr_bottom' else fixed
                ends.append(g)
            U = torch.cat([ends[0], U, ends[1]], dim=ax)
        return U

    def filled(self, U, t):
        """Every level with ghosts: a patch's own cells, else limited-linear values of the level below."""
        out = []
        for l in range(self.L):
            V = U[l] if l == 0 else torch.where(self.has[l], U[l], self.prolonged(out[l - 1], l))
            out.append(self.padded(V, l, t))
        return out

    def inner(self, A, ax=None, start=0, n=0):
        """Interior of a padded array, or a window of it along axis ax."""
        for a in range(1, self.dim + 1):
            A = A.narrow(a, start, n) if a == ax else A.narrow(a, G, A.shape[a] - 2 * G)
        return A

    def prolonged(self, A, l):
        C = self.inner(A)
        slopes = []
        for d in range(self.dim):
            ax = self.dim - d
            n = C.shape[ax]
            a, b = self.inner(A, ax, G + 1, n) - C, C - self.inner(A, ax, G - 1, n)
            slopes.append(torch.where(a * b <= 0, 0.0, torch.where(a.abs() <= b.abs(), a, b)))
        kids = []
        ok = None
        for k in range(1 << self.dim):
            v = C
            for d in range(self.dim):
                v = v + 0.25 * slopes[d] if k >> d & 1 else v - 0.25 * slopes[d]
            good = (v[0] > 0) & (_primitives(v, self.dim, self.gamma)[1] > 0)
            ok = good if ok is None else ok & good
            kids.append(v)
        out = torch.empty([self.dim + 2] + self.n[l][::-1], dtype=torch.float64, device='cuda')
        for k, v in enumerate(kids):
            at = tuple(slice(k >> d & 1, None, 2) for d in reversed(range(self.dim)))
            out[(slice(None),) + at] = torch.where(ok, v, C)
        return out

    def fluxes(self, A, l):
        """Face values of a level along every dimension, in global variable order."""
        dim, gamma, flux = self.dim, self.gamma, self.w['flux']
        u, p, T = _primitives(A, dim, gamma)
        out = []
        for d in range(dim):
            ax, n = dim - d, self.n[l][d]
            tang = [e for e in range(dim) if e != d]
            cut = lambda f, s, m: self.inner(f.unsqueeze(0), ax, s, m)[0]    # noqa: E731
            nodes = lambda f, s, k, m: [cut(f, s + j, m) for j in range(k)]    # noqa: E731
            pencils = lambda s, k, m: (nodes(p, s, k, m), nodes(u[d], s, k, m), [nodes(u[e], s, k, m) for e in tang],   # noqa: E731
                                       nodes(T, s, k, m))
            if flux in ('rusanov', 'hllc'):
                F = _weno_flux(*pencils(0, 6, n + 1), gamma, flux == 'hllc')
            else:
                Fc = _central_flux(*pencils(0, 4, n + 3), gamma)
                F = [(26 * f.narrow(ax - 1, 1, n + 1) - f.narrow(ax - 1, 0, n + 1) - f.narrow(ax - 1, 2, n + 1)) / 24 for f in Fc]
            if flux == 'hybrid':
                th, shock = self.w['theta_switch'], False
                rho = p / T
                for f in (rho, p):
                    q = nodes(f, 0, 6, n + 1)
                    for k in range(1, 5):
                        shock = shock | ((q[k + 1] - q[k - 1]).abs() > th * (q[k + 1] + 2 * q[k] + q[k - 1]))
                F = [torch.where(shock, a, b) for a, b in zip(_weno_flux(*pencils(0, 6, n + 1), gamma, False), F)]
            order = [0] + [1 if e == d else 2 + tang.index(e) for e in range(dim)] + [dim + 1]
            out.append(torch.stack([F[k] for k in order]))
        return out

    def corrected(self, F, fine, l):
        """Coarse faces between a leaf cell and a covered one take the mean of the fine faces."""
        for d in range(self.dim):
            ax = self.dim - d
            n = self.n[l][d]
            c = self.cov[l].unsqueeze(0)
            per = self.w['bc'][d][0] == 'periodic'
            no = torch.zeros_like(c.narrow(ax, 0, 1))
            c = torch.cat([c.narrow(ax, n - 1, 1) if per else no, c, c.narrow(ax, 0, 1) if per else no], dim=ax)
            h = self.has[l].unsqueeze(0)
            h = torch.cat([h.narrow(ax, n - 1, 1) if per else no, h, h.narrow(ax, 0, 1) if per else no], dim=ax)
            leaf = h & ~c
            here = (c.narrow(ax, 0, n + 1) & leaf.narrow(ax, 1, n + 1)) | (c.narrow(ax, 1, n + 1) & leaf.narrow(ax, 0, n + 1))
            f = fine[d]
            f = f.index_select(ax, torch.arange(0, f.shape[ax], 2, device='cuda'))
            for e in range(self.dim):
                if e != d:
                    b = self.dim - e
                    k = torch.arange(0, f.shape[b], 2, device='cuda')
                    f = 0.5 * (f.index_select(b, k) + f.index_select(b, k + 1))
            F[d] = torch.where(here, f, F[d])
        return F

    def restricted(self, U):
        for l in range(self.L - 1, 0, -1):
            m = U[l]
            for ax in range(1, self.dim + 1):
                k = torch.arange(0, m.shape[ax], 2, device='cuda')
                m = 0.5 * (m.index_select(ax, k) + m.index_select(ax, k + 1))
            U[l - 1] = torch.where(self.cov[l - 1], m, U[l - 1])
        return U

    def cfl(self, U):
        lam = 0.0
        for l in range(self.L):
            leaf = self.has[l] & ~self.cov[l]
            V = U[l][:, leaf]
            if V.numel():
                u, p, T = _primitives(V, self.dim, self.gamma)
                c = torch.sqrt(self.gamma * T)
                lam = max(lam, float(sum((u[d].abs() + c) / self.dx[l][d] for d in range(self.dim)).max()))
        return self.w['cfl'] / lam


def _dmr_states(gamma):
    r1, p1, M = 1.4, 1.0, 10.0
    r2 = r1 * (gamma + 1) * M * M / ((gamma - 1) * M * M + 2)
    p2 = p1 * (2 * gamma * M * M - (gamma - 1)) / (gamma + 1)
    v = M * math.sqrt(gamma * p1 / r1) * (1 - r1 / r2)
    out = []
    for r, a, b, p in ((r1, 0.0, 0.0, p1), (r2, v * math.sqrt(3) / 2, -v / 2, p2)):
        out.append([torch.tensor(x, dtype=torch.float64, device='cuda') for x in (r, r * a, r * b, p / (gamma - 1) + 0.5 * r * (a * a + b * b))])
    return out


def _advance64(w, levels, coords, data, steps):
    """SSP-RK3 steps of the whole hierarchy, all levels with the same dt."""
    H = _Dense64(w, levels, coords)
    U0, t = H.dense(levels, data), 0.0
    for _ in range(steps):
        dt = H.cfl(U0)
        U = U0
        for a, b, tf in ((0.0, 1.0, 0.0), (0.75, 0.25, 1.0), (1 / 3, 2 / 3, 0.5)):
            A = H.filled(U, t + tf * dt)
            new, fine = [None] * H.L, None
            for l in reversed(range(H.L)):
                F = H.fluxes(A[l], l)
                if fine is not None:
                    F = H.corrected(F, fine, l)
                V = U[l]
                for d in range(H.dim):
                    ax = H.dim - d
                    V = V - dt / H.dx[l][d] * (F[d].narrow(ax, 1, H.n[l][d]) - F[d].narrow(ax, 0, H.n[l][d]))
                new[l] = torch.where(H.has[l] & ~H.cov[l], a * U0[l] + b * V, U[l])
                fine = F
            U = H.restricted(new)
        U0, t = U, t + dt
    return H.patches(U0)
