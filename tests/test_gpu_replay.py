"""opts.graphs on levels above the size that runs as one kernel: the repeated
passes are replayed from one captured graph, with the results of the launches
it recorded."""
import numpy as np
import pytest

import graphgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2608_01503_gb300 as lc  # noqa: E402


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.fixture(scope="module")
def graphs():
    out = {"rmat": gg.rmat(18, seed=7), "grid": gg.grid_cpm(side=100)}
    assert all(g.n + g.nnz > 4_000_000 for g in out.values())
    return out


def replayed(res, plain):
    """Passes that were replayed: a captured pass counts the kernel that loads its
    temperature in the class "apply", a direct one in "other"."""
    return res["kernel_launches"]["apply"] - plain["kernel_launches"]["apply"]


@pytest.mark.parametrize("stream", ["current", "default", "own"])
@pytest.mark.parametrize("name", ["rmat", "grid"])
def test_one_graph(graphs, name, stream):
    g = graphs[name]
    args = (dev(g.row_ptr), dev(g.col), dev(g.ew), dev(g.vw), g.lam_num, g.lam_den)
    s = {"current": None, "default": torch.cuda.default_stream(), "own": torch.cuda.Stream()}[stream]
    torch.cuda.synchronize()
    want, plain = lc.lc_cluster(*args)
    got, res = lc.lc_cluster(*args, opts=lc.Options(graphs=True), stream=s)
    torch.cuda.synchronize()
    assert torch.equal(got, want) and res["phi"] == plain["phi"]
    # level 0: four of six passes from singletons, five of six on the way back
    assert replayed(res, plain) >= 9


def test_batch(graphs):
    p = gg.pack([graphs["grid"], gg.sbm_planted(n=3000, blocks=30, p_in=0.05, p_out=0.002, seed=8), gg.rmat(15, seed=9)])
    args = (dev(p["row_ptr"]), dev(p["col"]), dev(p["ew"]), dev(p["vw"]), p["graph_ptr"], p["lam_num"], p["lam_den"])
    want, plain = lc.lc_cluster_batch(*args)
    got, res = lc.lc_cluster_batch(*args, opts=lc.Options(graphs=True))
    assert torch.equal(got, want) and [r["phi"] for r in res] == [r["phi"] for r in plain]
    assert replayed(res[0], plain[0]) >= 9
