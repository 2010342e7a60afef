"""First calls of a process: a kernel whose dynamic and static shared memory together pass
48 KB by a little needs its limit raised before its first launch (a block of 100
functions stages 49052 bytes and 128 more).  A process of its own for each, so that no
other call has raised it earlier."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

PROGRAM = """
import sys
sys.path.insert(0, {root!r})
import numpy as np, torch
import paper_2004_10811_gb300 as pkg
n = {n}
rng = np.random.default_rng(n)
q, _ = np.linalg.qr(rng.standard_normal((n, n)))
w = np.where(np.arange(n) < n // 3, -1.0, 1.0) * (0.3 + 0.7 * rng.random(n))
a = (q * w) @ q.T
a = (a + a.T) / 2
K = torch.from_numpy(a.ravel().copy()).cuda()
with pkg.Plan(np.array([n], np.int32), np.array([0, 1], np.int64), np.array([0], np.int32), prec={prec!r}) as plan:
    D = plan.sign(K, 0.0).cpu().numpy().reshape(n, n)
assert np.max(np.abs(D - (q * (w < 0)) @ q.T)) <= {tol}, n
print("all")
"""


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("mixed", 1e-7), ("fp32", 1e-4)])
@pytest.mark.parametrize("n", [100, 161])
def test_one_block(n, prec, tol):
    import __graft_entry__ as g
    g.build()
    r = subprocess.run([sys.executable, "-c", PROGRAM.format(root=g.ROOT, n=n, prec=prec, tol=tol)],
                       capture_output=True, text=True, timeout=300)
    assert r.stdout.strip().endswith("all"), r.stderr[-2000:]
