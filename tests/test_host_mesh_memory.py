"""The host mesh holds one byte per position that a patch can have: the peak
memory of a process that closes a mesh of 50 million positions (48 x 48 base
patches, eight levels) grows by less than 1.5 bytes per position and 16 MB.
Beyond 2^26 positions it keeps a hash set instead, with the same results as the
oracle's hierarchy rules."""
import os
import random
import subprocess
import sys

from oracle.mesh import Mesh, canon

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = '''
import resource
import numpy as np
from paper_2508_05020_gb300 import amr
base, levels = 48, 8
keys = [(0, x, y, 0) for y in range(base) for x in range(base)]
amr.mesh_close(2, (2, 2), (0, 0), 1, [(0, x, y, 0) for y in range(2) for x in range(2)])
before = resource.getrusage(resource.RUSAGE_SELF).ru_maxrss
out, created, deleted = amr.mesh_close(2, (base, base), (0, 0), levels - 1, keys, refine=[(0, 5, 5, 0)])
assert (len(out), created, deleted) == (base * base + 4, 4, 0)
print(resource.getrusage(resource.RUSAGE_SELF).ru_maxrss - before)
'''


def test_mesh_takes_one_byte_per_position():
    r = subprocess.run([sys.executable, '-c', CODE], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    positions = sum((48 << l) ** 2 for l in range(8))
    assert int(r.stdout) * 1024 < 1.5 * positions + (16 << 20), r.stdout


def test_more_positions_than_the_dense_array_takes():
    from paper_2508_05020_gb300 import amr
    rows = lambda keys: [[l, *c] for l, c in sorted(keys, key=canon)]   # noqa: E731
    base, top = (72, 72), 7                              # 113 million positions
    rng = random.Random(5)
    m = Mesh(2, base, (True, False), top)
    changed = 0
    for _ in range(25):
        near = [k for k in m.patches if m.is_leaf(k) and k[0] < top and k[1][0] < 3 << k[0] and k[1][1] < 3 << k[0]]
        req = rng.sample(sorted(near, key=canon), 2)
        cand = [k for k in sorted(m.patches, key=canon) if m.has_children(k) and rng.random() < 0.3]
        got, n_created, n_deleted = amr.mesh_close(2, base, (True, False), top, rows(m.patches), rows(req), rows(cand))
        created = m.refine(req)
        deleted = m.coarsen(cand, created)
        assert got.tolist() == rows(m.patches)
        assert (n_created, n_deleted) == (len(created), len(deleted))
        changed += bool(deleted)
    assert changed >= 5 and max(k[0] for k in m.patches) >= 3
