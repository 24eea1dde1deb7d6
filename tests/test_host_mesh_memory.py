"""The host mesh holds one byte per position that a patch can have: the peak
memory of a process that closes a mesh of 50 million positions (48 x 48 base
patches, eight levels) grows by less than 1.5 bytes per position and 16 MB."""
import subprocess
import sys

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
    import os
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, '-c', CODE], cwd=root, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    positions = sum((48 << l) ** 2 for l in range(8))
    assert int(r.stdout) * 1024 < 1.5 * positions + (16 << 20), r.stdout
