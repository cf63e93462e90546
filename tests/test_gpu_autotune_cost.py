"""What a call with new sizes pays for the choice of a tile: at most three timed products per candidate
and twelve more for those that come near the best (the autotuner's log, in a process of its own)."""
import os
import re
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = """
import sys, torch, synth
import paper_2306_12616_gb300 as fo
s = fo.Solver(0)
n = int(sys.argv[1])
h = torch.from_numpy(synth.tight_binding(n, 3)).to("cuda:0")
p, r = s.density_matrix(h, n / 2, s.params(60, 0.1, precision="bf16x3"))
print("TILE", r["tile_n"], r["tile_ctas"], r["tile_drain"], r["tile_store"])
"""


@pytest.mark.parametrize("n", [64, 1000, 3000])
def test_products_timed(n):
    env = dict(os.environ, FERMI_AUTOTUNE_LOG="1")
    out = subprocess.run([sys.executable, "-c", PROGRAM, str(n)], cwd=ROOT, env=env, capture_output=True, text=True,
                         check=True)
    runs = re.findall(r"tile (\d+)x(\d+)x(\d+) store (\d) persistent \d: ([\d.]+) ms per product \((\d+)\)", out.stderr)
    times = {}
    for *tile, ms, reps in runs:
        times.setdefault(tuple(map(int, tile)), []).append((float(ms), int(reps)))
    assert len(times) == 10
    assert all(len(v) <= 2 and v[0][1] == 3 and v[-1][1] <= 12 for v in times.values())
    # the fastest is the one used
    used = tuple(int(x) for x in re.search(r"TILE (\d+) (\d+) (\d+) (\d+)", out.stdout).groups())
    assert min(m for m, _ in times[used]) == min(m for v in times.values() for m, _ in v)
