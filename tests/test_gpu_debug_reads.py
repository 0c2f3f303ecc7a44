"""The debug library's range checks of the slot reads in the far-field kernels.  The float64 one-sided kernel's
writes are not checked, so that a shrunken limit refuses reads alone: all of them, or all but the first tile's first
slot.  Either way the evaluation reports PSUM_ERR_INTERNAL and every output is NaN, the points of the allowed slot too;
the next evaluation on the same context is exact.  Run in a child process, which loads the debug library."""
import json
import os
import subprocess
import sys

import pytest

from paper_1310_4374_gb300 import binding as B

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

_SCRIPT = r"""
import json, sys
import torch
sys.path.insert(0, sys.argv[1])
from paper_1310_4374_gb300 import binding as B
from paper_1310_4374_gb300 import workloads as W
out = {"checks": B.psum_debug_checks(), "cases": []}
s = W.config(1)
x = torch.as_tensor(s.x, dtype=torch.float64, device="cuda")
q = torch.as_tensor(s.q, dtype=torch.float64, device="cuda")
y = (0.75 * x[:301]).contiguous()
pc = B.PeriodicCoulomb(s.d, s.p, s.M, precision="fp64", pairs="one-sided")
def run(call, phi, g):
    if call == "points":
        B.psum_eval_points(pc.plan, x, q, y, phi, g)
    else:
        B.psum_eval(pc.plan, x, q, phi, g)
    return B.psum_sync(pc.plan)
for call in ("eval", "points"):
    for grad in (True, False):
        n = y.shape[0] if call == "points" else q.numel()
        new = lambda: (torch.zeros(n, dtype=torch.float64, device="cuda"),
                       torch.zeros((n, 3), dtype=torch.float64, device="cuda") if grad else None)
        a = new()
        ok = run(call, *a)
        for limit in (256, 512):
            B.psum_debug_bounds_limit(pc.plan, limit)
            b = new()
            st = run(call, *b)
            nan = all(bool(torch.isnan(t).all()) for t in b if t is not None)
            B.psum_debug_bounds_limit(pc.plan, 0)
            c = new()
            again = run(call, *c)
            same = all(bool(torch.equal(u, v)) for u, v in zip(a, c) if u is not None)
            out["cases"].append([call, grad, limit, ok, st, nan, again, same])
pc.close()
print(json.dumps(out))
"""


def test_refused_reads_are_reported():
    from paper_1310_4374_gb300 import build as _b
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, PSUM_LIB=_b.build(debug=True))
    r = subprocess.run([sys.executable, "-c", _SCRIPT, root], env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    out = json.loads(r.stdout.strip().splitlines()[-1])
    assert out["checks"] is True and len(out["cases"]) == 8
    for call, grad, limit, ok, st, nan, again, same in out["cases"]:
        assert ok == again == B.PSUM_OK and same, (call, grad, limit, ok, again, same)
        assert st == B.PSUM_ERR_INTERNAL and nan, (call, grad, limit, st, nan)
