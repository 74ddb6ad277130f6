"""Ends of small levels at the sizes where the second kernel's work changes
hands: slot runs of 256 to 2,048, several runs a warp, coarse rows that cross
many runs, one block and many; labels, levels and objective equal those of the
separate kernels (Options(profile=True))."""
import numpy as np
import pytest

import graphgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2608_01503_gb300 as lc  # noqa: E402


def blocks(n, k, degree, seed):
    """A block model of n vertices; half of the degree leaves the block."""
    return gg.sbm_planted(n=n, blocks=k, p_in=min(1.0, degree / 2 / (n / k)), p_out=degree / 2 / n, seed=seed)


GRAPHS = {
    "a block of threads": lambda: blocks(60, 3, 8, 1),
    "runs of 256": lambda: blocks(3000, 30, 12, 2),
    "runs of 512": lambda: blocks(40_000, 60, 14, 3),
    "runs of 1,024 and more": lambda: gg.rmat(16, seed=4),
    "several runs a warp": lambda: blocks(20_000, 200, 190, 5),
    "few coarse rows": lambda: blocks(12_000, 2, 120, 6),
    "nothing merges for long": lambda: gg.cpm_inputs(*gg.rmat_csr(14, seed=7), 1, 2),
    "lattice, many levels": lambda: gg.grid_cpm(side=60),
}


@pytest.mark.parametrize("name", list(GRAPHS))
def test_levels_equal_the_separate_kernels(name):
    g = GRAPHS[name]()
    assert g.n + g.nnz <= 4_000_000
    args = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (g.row_ptr, g.col, g.ew, g.vw)]
    lam = (g.lam_num, g.lam_den)
    for call in (lc.lc_cluster, lc.lc_cluster_leiden):
        a, ra = call(*args, *lam)
        b, rb = call(*args, *lam, opts=lc.Options(profile=True))
        assert torch.equal(a, b)
        assert all(ra[k] == rb[k] for k in ("phi", "levels", "n_clusters", "passes_total"))


def test_batch_whose_graphs_end_at_different_levels():
    pool = [GRAPHS[k]() for k in ("a block of threads", "runs of 256", "nothing merges for long")] + \
           [gg.grid_cpm(side=20), blocks(500, 2, 6, 8), gg.rmat(12, seed=9)]
    p = gg.pack(pool)
    args = [torch.from_numpy(np.ascontiguousarray(p[k])).cuda() for k in ("row_ptr", "col", "ew", "vw")]
    rest = (p["graph_ptr"], p["lam_num"], p["lam_den"])
    a, ra = lc.lc_cluster_batch(*args, *rest)
    b, rb = lc.lc_cluster_batch(*args, *rest, opts=lc.Options(profile=True))
    assert torch.equal(a, b)
    assert [(x["phi"], x["levels"], x["n_clusters"]) for x in ra] == [(x["phi"], x["levels"], x["n_clusters"]) for x in rb]
    assert len({x["levels"] for x in ra}) > 2
