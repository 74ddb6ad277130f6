"""Bin plans and the one-kernel passes of small levels: a plan that gives blocks
short rows runs as separate kernels, and a level's end does not take its hub
rows one after the other."""
import statistics
import time

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


def run(g, **kw):
    return lc.lc_cluster(dev(g.row_ptr), dev(g.col), dev(g.ew), dev(g.vw), g.lam_num, g.lam_den, opts=lc.Options(**kw))


@pytest.mark.parametrize("bins,fused", [
    ((), True),
    ((8, 16, 32, 128, 256, 256, 256, 256, 256), True),
    ((8, 16, 32, 128, 128, 128, 256, 2048, 4096), True),
    ((8, 16, 32, 128, 255, 255, 255, 2048, 4096), False),
    ((8, 16, 32, 64, 127, 512, 1024, 2048, 4096), False),
    ((8,) * 9, False),
])
def test_short_rows_of_blocks_run_as_separate_kernels(bins, fused):
    g = gg.sbm_planted(n=4000, blocks=40, p_in=0.06, p_out=0.002, seed=4)
    labels, res = run(g, bins=bins)
    want, separate = run(g, bins=bins, profile=True)
    assert torch.equal(labels, want) and res["phi"] == separate["phi"]
    few, many = (sum(r["kernel_launches"].values()) for r in (res, separate))
    assert (2 * few < many) if fused else (few == many)


@pytest.mark.parametrize("chunk", [0, 256])
def test_thousands_of_one_chunk_hubs(chunk):
    """Every row above 8 edges a hub: more hubs than the plan's one block cuts,
    most of one chunk and settled by a lane, a few of many; from singletons,
    from labels with movers to new clusters, in a batch and with pLeiden."""
    rp, col, ew = gg.rmat_csr(15, seed=6)
    assert (np.diff(rp) > 8).sum() > 8192
    plan = dict(bins=(8,) * 9, hub_chunk=chunk)
    for g in (gg.modularity_inputs(rp, col, ew), gg.cpm_inputs(rp, col, ew, 1, 3)):
        args = (dev(g.row_ptr), dev(g.col), dev(g.ew), dev(g.vw), g.lam_num, g.lam_den)
        start = dev(gg.random_labels(g.n, 40, seed=3))
        for call in (lc.lc_cluster, lc.lc_cluster_leiden, lambda *a, **k: lc.lc_local_move(*a, start.clone(), **k)):
            a, ra = call(*args)
            b, rb = call(*args, opts=lc.Options(**plan))
            assert torch.equal(a, b) and ra["phi"] == rb["phi"]
    p = gg.pack([gg.modularity_inputs(rp, col, ew), gg.rmat(11, seed=5), gg.grid_cpm(side=12)])
    args = [dev(p[k]) for k in ("row_ptr", "col", "ew", "vw")] + [p["graph_ptr"], p["lam_num"], p["lam_den"]]
    a, ra = lc.lc_cluster_batch(*args)
    b, rb = lc.lc_cluster_batch(*args, opts=lc.Options(**plan))
    assert torch.equal(a, b) and [r["phi"] for r in ra] == [r["phi"] for r in rb]


def test_hub_rows_of_a_small_level_end_at_once():
    """Every row above 256 entries a hub: 974 of them on this graph.  Taken
    one after the other they made the call 4.5 times as long."""
    g = gg.rmat(16, seed=3)

    def ms(**kw):
        args = (dev(g.row_ptr), dev(g.col), dev(g.ew), dev(g.vw), g.lam_num, g.lam_den)
        times = []
        for _ in range(12):
            torch.cuda.synchronize()
            t = time.perf_counter()
            labels, _ = lc.lc_cluster(*args, opts=lc.Options(**kw))
            times.append(time.perf_counter() - t)
        return statistics.median(times[2:]), labels

    default, a = ms()
    hubs, b = ms(bins=(8, 16, 32, 128, 256, 256, 256, 256, 256))
    assert torch.equal(a, b)
    assert hubs < 2.5 * default
