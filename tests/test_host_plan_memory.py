"""Host memory of a plan of wide operators: the fused matrices in FP32, once more
while their vector moves as it grows, and no FP64 copies of matrices that no
group pass takes (twice as much again).  In a process of its own, by its peak
resident size."""
import subprocess
import sys

import pytest

SCRIPT = """
import resource
import numpy as np
import workloads as W
import paper_2608_16940_gb300 as q
n, count = %d, 1500
u = W.haar_unitary(64, np.random.default_rng(0))
ops = q.OpArray([W.Op(tuple(range(i %% 8, i %% 8 + 6)), u) for i in range(count)])
before = resource.getrusage(resource.RUSAGE_SELF).ru_maxrss
p = q.qsa_plan_create(ops, n, q.make_opts(planner=%s, kmax=6))
after = resource.getrusage(resource.RUSAGE_SELF).ru_maxrss
print((after - before) * 1024 / (count * 2 * 4096 * 4))
"""


@pytest.mark.parametrize("n,planner", [(20, "q.QSA_PLAN_PER_GATE"), (20, "q.QSA_PLAN_GREEDY"), (27, "q.QSA_PLAN_GREEDY")])
def test_wide_plans_hold_no_double_copies(n, planner):
    import __graft_entry__
    __graft_entry__._build_module().build()
    out = subprocess.run([sys.executable, "-c", SCRIPT % (n, planner)], capture_output=True, text=True,
                         cwd=__graft_entry__.ROOT, timeout=300)
    assert out.returncode == 0, out.stderr[-2000:]
    assert float(out.stdout) <= 2.2   # times the FP32 matrices
