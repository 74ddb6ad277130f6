"""What a call on a graph of few vertices takes is sized by the graph: limits
that were enough before the cooperative kernels had scratch of their own still
are."""
import numpy as np
import pytest

import graphgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2608_01503_gb300 as lc  # noqa: E402


@pytest.mark.parametrize("n,cluster,leiden,move", [(20, 7945, 14141, 7189), (100, 38721, 63193, 37825),
                                                   (1000, 424817, 699617, 378477)])
def test_limits_of_small_graphs(n, cluster, leiden, move):
    g = gg.sbm_planted(n=n, blocks=n // 20, p_in=8 / 20, p_out=4 / n, seed=1)
    args = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (g.row_ptr, g.col, g.ew, g.vw)]
    lam = (g.lam_num, g.lam_den)
    lc.lc_cluster(*args, *lam, opts=lc.Options(scratch_limit=cluster))
    lc.lc_cluster_leiden(*args, *lam, opts=lc.Options(scratch_limit=leiden))
    lc.lc_local_move(*args, *lam, torch.zeros(n, dtype=torch.int32, device="cuda"), opts=lc.Options(scratch_limit=move))
