"""FP64 roundings whose digit scratch is refused run on the FP64 units: an
allocator that serves every request up to a limit between the cores (67 MB
here) and the digits of the tall factors (240 MB): in all three roundings, after
the scratch has grown once, and until the last one.  At tol = 0 the tensor comes back: the 1e-12 of the
other FP64 rounding tests.  Fresh processes: the allocator may only change
while no context or tensor exists."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import numpy as np, torch
from paper_2403_04946_gb300 import binding as B
from oracle import tt
import synthetic
limits = {limits}  # MB, per rounding
dev = torch.cuda.current_device()
state = dict(limit=0, refused=0)
def alloc(nb):
    if nb > state["limit"] << 20:
        state["refused"] += 1
        return 0
    return torch.cuda.caching_allocator_alloc(nb, dev)
B.hopf_set_allocator(alloc, lambda p: torch.cuda.caching_allocator_delete(p))
state["limit"] = limits[0]
d, n = 5, 64
big = [1, 64, 256, 256, 64, 1]
ctx = B.Context(d=d, n=n, nu=0.02, tol=0.0, rank_cap=256, L=4.0)
err = []
for limit, ranks in zip(limits, ([1, 48, 48, 48, 40, 1], big, big)):
    state["limit"] = limit
    x = synthetic.random_tt_cores(d, n, ranks, seed=5)
    t = ctx.tt_from_host(x, max_rank=256)
    ctx.tt_round(t, 0.0, 256, forced_ranks=ranks)
    err.append(tt.diff_norm(ctx.tt_to_host(t), x) / tt.norm(x))
    ctx.tt_free(t)
ctx.close()
B.hopf_set_allocator(None, None)
print(max(err), state["refused"])
"""


@pytest.mark.parametrize("limits", [(150, 150, 150), (2000, 150, 150), (150, 150, 2000)])
def test_refused_scratch_falls_back(limits):
    r = subprocess.run([sys.executable, "-c", CODE.format(limits=limits)], cwd=ROOT, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    err, refused = r.stdout.split()
    assert float(err) < 1e-12
    assert int(refused) > 0
