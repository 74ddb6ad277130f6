"""The one-kernel LocalMovePasses of small levels against the oracle and the
separate kernels (Options(profile=True) runs those): the row lengths where
its work changes hands, hub rows beyond a block's table, new clusters,
batches, and single-pass calls.  Everything is integer and must be equal."""
import numpy as np
import pytest

import graphgen as gg
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2608_01503_gb300 as lc  # noqa: E402


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def stars(degrees, extra=3, seed=0):
    """A star per degree, the leaves joined by a few random edges."""
    rng = np.random.default_rng(seed)
    n = len(degrees) + sum(degrees)
    src, dst, at = [], [], len(degrees)
    for k, d in enumerate(degrees):
        leaves = np.arange(at, at + d)
        src.append(np.full(d, k))
        dst.append(leaves)
        at += d
    m = extra * len(degrees) * 100
    src.append(rng.integers(0, n, m))
    dst.append(rng.integers(0, n, m))
    s, t = np.concatenate(src), np.concatenate(dst)
    keep = s != t
    return gg.from_edges(n, s[keep], t[keep], seed=seed, wmin=1, wmax=8)


def graphs():
    edge = stars([7, 8, 9, 15, 16, 17, 31, 32, 33, 127, 128, 129, 255, 256, 257, 511, 513, 1023, 1025, 2049, 4096])
    big = stars([4097, 8191, 8192, 8193, 20000], seed=1)
    return {
        "bin edges, modularity": gg.modularity_inputs(*edge),
        "bin edges, CPM 1/3": gg.cpm_inputs(*edge, 1, 3),
        "hubs around a block's table": gg.modularity_inputs(*big),
        "hubs, CPM 1/2": gg.cpm_inputs(*big, 1, 2),
        "one vertex": gg.cpm_inputs(np.zeros(2, np.int64), np.zeros(0, np.int32), np.zeros(0, np.int32), 1, 2),
        "edgeless": gg.cpm_inputs(np.zeros(1001, np.int64), np.zeros(0, np.int32), np.zeros(0, np.int32), 1, 2),
        "lattice": gg.grid_cpm(side=13),
        "rmat": gg.rmat(13, seed=4),
    }


@pytest.mark.parametrize("name", list(graphs()))
@pytest.mark.parametrize("passes", [1, 2, 6])
def test_clustering_equals_oracle_and_separate_kernels(name, passes):
    g = graphs()[name]
    args = (dev(g.row_ptr), dev(g.col), dev(g.ew), dev(g.vw), g.lam_num, g.lam_den)
    phi = [(3, 4)] * 4 + [(1, 4)] * 2
    a, ra = lc.lc_cluster(*args, opts=lc.Options(pass_limit=passes))
    b, rb = lc.lc_cluster(*args, opts=lc.Options(pass_limit=passes, profile=True))
    ref, orc, _ = oracle.louvain_plus(g, oracle.Params(pass_limit=passes, phi=phi))
    assert np.array_equal(a.cpu().numpy(), ref) and ra["phi"] == orc["phi"]
    assert torch.equal(a, b) and ra["phi"] == rb["phi"]
    # far fewer kernels in the fused call: it did take that path
    assert sum(ra["kernel_launches"].values()) < sum(rb["kernel_launches"].values())


@pytest.mark.parametrize("lam", [(1, 2), (1, 50)])
def test_local_move_from_a_clustering_with_new_clusters(lam):
    """Random labels under a strong CPM: many movers to new empty clusters."""
    g = gg.cpm_inputs(*gg.rmat_csr(12, seed=7), *lam)
    start = gg.random_labels(g.n, 40, seed=3)
    args = (dev(g.row_ptr), dev(g.col), dev(g.ew), dev(g.vw), g.lam_num, g.lam_den)
    a, ra = lc.lc_local_move(*args, dev(start).clone())
    b, rb = lc.lc_local_move(*args, dev(start).clone(), opts=lc.Options(profile=True))
    assert torch.equal(a, b) and ra["phi"] == rb["phi"]
    out = oracle.local_move(g, start)
    assert np.array_equal(a.cpu().numpy(), out[0] if isinstance(out, tuple) else out["labels"])


def test_batch_of_mixed_graphs():
    pool = [g for g in graphs().values() if g.nnz > 0] + \
           [gg.sbm_planted(n=300 + 50 * k, blocks=5, p_in=0.1, p_out=0.01, seed=k) for k in range(5)]
    p = gg.pack(pool)
    labels, res = lc.lc_cluster_batch(dev(p["row_ptr"]), dev(p["col"]), dev(p["ew"]), dev(p["vw"]), p["graph_ptr"],
                                      p["lam_num"], p["lam_den"])
    got = labels.cpu().numpy()
    for k, g in enumerate(pool):
        ref, orc, _ = oracle.louvain_plus(g)
        lo, hi = p["graph_ptr"][k], p["graph_ptr"][k + 1]
        assert np.array_equal(got[lo:hi], ref) and res[k]["phi"] == orc["phi"], k


@pytest.mark.parametrize("lam", [(1, 60_000), (7, 200_003), (1, 1_000_003)])
def test_gains_on_both_sides_of_32_bits(lam):
    """Edge weights up to 2^15 under lambda denominators that take the gains,
    their differences and the epsilon buckets' operands across 2^31 and 2^32,
    where the 32-bit forms hand over."""
    n, m = 1500, 12_000
    rng = np.random.default_rng(9)
    s, t = rng.integers(0, n, m), rng.integers(0, n, m)
    g = gg.cpm_inputs(*gg.from_edges(n, s[s != t], t[s != t], seed=9, wmin=1, wmax=1 << 15), *lam)
    args = (dev(g.row_ptr), dev(g.col), dev(g.ew), dev(g.vw), g.lam_num, g.lam_den)
    a, ra = lc.lc_cluster(*args)
    b, rb = lc.lc_cluster(*args, opts=lc.Options(profile=True))
    ref, orc, _ = oracle.louvain_plus(g)
    assert np.array_equal(a.cpu().numpy(), ref) and ra["phi"] == orc["phi"]
    assert torch.equal(a, b) and ra["phi"] == rb["phi"]
