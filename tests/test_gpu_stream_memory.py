"""Device memory that the level order's preparation takes at its peak, per edge.

The stream-ordered pool keeps what it reserved, so the device's free memory after the first preparation
of a process shows the peak.  The streams' sort needs the most: 48 bytes an edge of keys and positions
next to 24 (28 weighted) of the streams and 16 of the leading classes' records and, until it goes, the class order, and
the loaded graph's 8 (20); 20 more for the sort's scratch and the pool's granularity.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHILD = """
import sys
sys.path.insert(0, sys.argv[1])
import numpy as np, torch
import synth, paper_2307_15969_gb300 as pkg
g = synth.workload('rmat18')
u, v = torch.from_numpy(g.u).cuda(), torch.from_numpy(g.v).cuda()
w = torch.from_numpy(np.random.default_rng(1).integers(1, 9, g.m).astype(np.float32)).cuda() if int(sys.argv[2]) else None
torch.cuda.synchronize()
free = torch.cuda.mem_get_info()[0]
h = pkg.lowd_load_graph(g.n, u, v, w)
pkg.lowd_iterate(h, 0, schedule=2)
torch.cuda.synchronize()
print("PEAK", (free - torch.cuda.mem_get_info()[0]) / g.m)
"""


@pytest.mark.parametrize("weighted", [0, 1])
def test_bytes_per_edge(weighted):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_15969_gb300 import build
    build.build()
    p = subprocess.run([sys.executable, "-c", CHILD, ROOT, str(weighted)], capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stderr[-2000:]
    peak = float(p.stdout.split("PEAK")[1])
    assert peak <= 8 + 12 * weighted + 24 + 4 * weighted + 16 + 48 + 20, peak
