"""Memory of a plan whose tiles are split over their sources: the segment sums of a
tile take its own segments x row groups.  A tile of up to 32 targets and 16
segments holds 16 x 32 sums of 8 bytes, 4 KB; with what else a leaf of such
targets has (lists of up to 100 entries, 16 tasks of 320 bytes each and as much
again while they are sorted) 20 KB is ample.  (Sums for 256 rows of every tile
took 32 KB by themselves.)"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import torch
from paper_2012_06925_gb300 import binding as B
from paper_2012_06925_gb300 import workloads as W
tgt, src, q = W.make_problem("uniform", 400000, 30000, seed=2, sources_kind="uniform")
t, s, q = (torch.from_numpy(a).cuda() for a in (tgt, src, q))
with B.Plan(t[:, :100].contiguous(), s, q, n=1, theta=0.7, N0=300, M0=30) as p:
    p.compute()
torch.cuda.synchronize()
free = torch.cuda.mem_get_info()[0]
with B.Plan(t, s, q, n=1, theta=0.7, N0=300, M0=30) as p:
    p.compute()
    torch.cuda.synchronize()
    used = free - torch.cuda.mem_get_info()[0]
    leaves = p.stats()["num_target_leaves"]
print("RESULT", used, leaves)
"""


def test_segment_sums_take_the_tiles_own_size():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, BLDTT_TASK_CHUNKS="1", PYTHONPATH=root)
    out = subprocess.run([sys.executable, "-c", CODE], cwd=root, env=env, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr[-2000:]
    used, leaves = (int(v) for v in out.stdout.split("RESULT")[1].split())
    assert leaves > 10000
    assert used <= 20 * 1024 * leaves, (used, leaves)
