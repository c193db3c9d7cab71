"""Host memory of the planner follows the distinct pairs of a batch, not its quartets."""
import subprocess
import sys

SCRIPT = """
import ctypes, resource
import numpy as np
from paper_2307_03452_gb300 import lx
n = 1000
sh = np.zeros(4 * n, lx.SHELL_DTYPE)
sh["l"], sh["nprim"], sh["prim_offset"] = 2, 1, np.arange(4 * n)
q = np.zeros(n * n, lx.QUARTET_DTYPE)
i, j = np.divmod(np.arange(n * n), n)
q["s"] = np.stack([2 * i, 2 * i + 1, 2 * n + 2 * j, 2 * n + 2 * j + 1], 1)
size = lambda m: lx.load().lx_eri_workspace_size(lx._ptr(sh), len(sh), lx._ptr(q), m, lx.LX_SOLID)
assert size(n) > 0
before = resource.getrusage(resource.RUSAGE_SELF).ru_maxrss
assert size(n * n) > 0
print(resource.getrusage(resource.RUSAGE_SELF).ru_maxrss - before)
"""


def test_size_query_of_a_million_quartets_over_2000_pairs():
    # 2,000 pairs are 64 kB of table; one slot of 16 bytes per quartet would be 16 MB
    r = subprocess.run([sys.executable, "-c", SCRIPT], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    assert int(r.stdout) < 16 * 1024, f"{r.stdout.strip()} kB"
