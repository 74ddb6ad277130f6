"""A grid barrier that a block never reaches: its wait gives up after a short
limit, the call returns LC_ERR_DEVICE whichever barrier it was, nothing of the
unfinished state is indexed out of range, and the next call is right.

The checked build skips the arrival of one block at the K-th barrier of a call
(LC_DEBUG_BARRIER=K:polls); a failed index check in such a call would show as
its error's detail.  Runs in a child process, which loads that build."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.slow]

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2608_01503_gb300 import _build  # noqa: E402

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import os
import numpy as np, torch
import graphgen as gg
import paper_2608_01503_gb300 as lc
assert lc.lc_debug_enabled()
DEVICE = 10
dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
arrays = lambda g: (dev(g.row_ptr), dev(g.col), dev(g.ew), dev(g.vw))
args = lambda g: (*arrays(g), g.lam_num, g.lam_den)
sbm = gg.sbm_planted(n=4000, blocks=40, p_in=0.06, p_out=0.002, seed=4)
# strong CPM from random labels: many movers to new clusters, in several blocks
cpm = gg.cpm_inputs(*gg.rmat_csr(14, seed=7), 1, 2)
start = dev(gg.random_labels(cpm.n, 40, seed=3))
hub = gg.modularity_inputs(*gg.rmat_csr(13, seed=2))
S, P, H = args(sbm), args(cpm), args(hub)
pk = gg.pack([sbm, gg.rmat(11, seed=5), gg.sbm_planted(n=900, blocks=9, p_in=0.1, p_out=0.01, seed=1)])
B = (dev(pk["row_ptr"]), dev(pk["col"]), dev(pk["ew"]), dev(pk["vw"]), pk["graph_ptr"], pk["lam_num"], pk["lam_den"])
lab = torch.arange(hub.n, dtype=torch.int32, device="cuda") // 16
O = lc.Options
def contract():
    r = lc.lc_contract(*H[:4], lab, int(lab[-1]) + 1)
    return r[0], r[3]
CALLS = {
    "cluster": lambda: lc.lc_cluster(*S),
    "separate": lambda: lc.lc_cluster(*P, opts=O(profile=True)),
    "new clusters": lambda: lc.lc_local_move(*P, start.clone()),
    "new clusters, separate": lambda: lc.lc_local_move(*P, start.clone(), opts=O(profile=True)),
    "hubs": lambda: lc.lc_cluster(*H, opts=O(bins=(8, 16, 32, 128, 256, 256, 256, 256, 256), hub_chunk=256)),
    "leiden": lambda: lc.lc_cluster_leiden(*S),
    "leiden, hubs": lambda: lc.lc_cluster_leiden(*H),
    "batch": lambda: lc.lc_cluster_batch(*B),
    "iterated": lambda: lc.lc_cluster_iterated(*S, 2),
    "tables": lambda: lc.lc_cluster(*H, opts=O(tables=1)),
    "symmetry": lambda: lc.lc_cluster(*S, opts=O(symmetry=2)),
    "no passes": lambda: lc.lc_cluster(*S, opts=O(pass_limit=0)),
    "contract": contract,
}
for name, call in CALLS.items():
    want = [t.clone() for t in call() if torch.is_tensor(t)]
    failed = ended = 0
    for k in list(range(1, 30)) + [int(30 * 1.12 ** i) for i in range(40)]:
        os.environ["LC_DEBUG_BARRIER"] = f"{k}:3000"
        try:
            call()
            ended += 1
        except lc.LCError as e:
            assert e.code == DEVICE and e.detail == 0, (name, k, e.code, e.detail)
            failed += 1
        del os.environ["LC_DEBUG_BARRIER"]
        got = [t for t in call() if torch.is_tensor(t)]
        assert all(torch.equal(a, b) for a, b in zip(got, want)), (name, k)
        if ended >= 2:  # the call has fewer barriers than that
            break
    assert failed > 0, name
    print(name, failed, ended, flush=True)
torch.cuda.synchronize()
print("barriers ok")
"""


def test_a_wait_that_runs_out_is_an_error_and_no_more():
    _build.build(debug=True)
    p = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env={**os.environ, "LC_DEBUG": "1"}, capture_output=True,
                       text=True, timeout=600)
    assert p.returncode == 0, p.stdout + p.stderr
    assert "barriers ok" in p.stdout
